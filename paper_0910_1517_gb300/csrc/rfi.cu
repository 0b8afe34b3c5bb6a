// rfi.cu -- RFI-flagging stage for sm_103a: per-patch median / MAD statistics and
// flags (Sec. 5, Eq. 3-4), and a small convolutional flagger trained and run by
// hand-written kernels (the FP16 flagger's forward pass is rfi_tc.cu's; the rest
// here are direct 3x3 convolutions over 16x16 output tiles, FP16
// weights and activations, FP32 accumulation, FP32 gradients, Adam on FP32
// master weights).  Every network kernel is templated on the type TA its weights
// and activations are kept in: __half for the flagger, float for the FP32 build
// (rfi_create_fp32) that checks the kernels' arithmetic against the FP64 oracle.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>

#include "../../include/corr.h"
#include "../../include/rfi.h"
#include "common.cuh"
#include "rfi_tc.cuh"

namespace gbx {
void set_last_error(const char* msg);
}

namespace {

__device__ __forceinline__ float ldf(const __half* p) { return __half2float(*p); }
__device__ __forceinline__ float ldf(const float* p) { return *p; }
// four consecutive values; `wide`: the address is aligned to all four
__device__ __forceinline__ float4 ldf4(const __half* p, bool wide) {
    if (!wide) return make_float4(ldf(p), ldf(p + 1), ldf(p + 2), ldf(p + 3));
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x)), b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float4 ldf4(const float* p, bool wide) {
    return wide ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
}
__device__ __forceinline__ void stf(__half* p, float v) { *p = __float2half_rn(v); }
__device__ __forceinline__ void stf(float* p, float v) { *p = v; }

constexpr int PH = 64, PW = 64, PHW = PH * PW;   // patch: 64 dumps x 64 channels
constexpr int T = 16, TH = T + 2;                 // output tile and tile with halo
constexpr int kTiles = (PH / T) * (PW / T);       // 16 tiles per patch
constexpr int NPAR = 9441;
constexpr int OW1 = 0, OB1 = 144, OW2 = 160, OB2 = 4768, OW3 = 4800, OB3 = 9408, OW4 = 9424, OB4 = 9440;

// ---------------------------------------------------------------- convolution
// A CTA computes a 16 x 32 output tile of one patch for all CO output channels: a thread takes two
// rows of four pixels and 8 channels, two channels a packed FP32x2 operation, input channel by input
// channel and tap by tap (24 window values and 18 16-byte weight reads serve 288 packed operations).
// MODE 0 (forward):       out[o] = relu(b[o] + sum_c sum_tap w[c][tap][o] in[c][pixel + tap])   (-> TA)
// MODE 1 (backward data): the same correlation without bias / ReLU on dZ = dA * (act > 0)        (fp32 -> fp32)
// w is laid out [CI][9][CO] so that one (c, tap) reads consecutive weights (a broadcast).
// TIN: type of the forward input (the FP16 patches for layer 1, TA after it); TA: weights and activations.
// What bounds it: the FP32 pipe, with the shared-memory reads of the weights (four cycles each, shared
// or not) close behind.  256 patches, backward data of layers 3 / 2: 0.24 / 0.25 ms; 0.33 / 0.43 ms with a
// pixel a thread (9 or 5 reads for 32 or 16 multiply-adds), no better with four.
constexpr int CTY = 16, CTX = 32, CPX = 36, CCK = 8;   // tile, row pitch with halo, input channels a round
constexpr int kCTiles = (PH / CTY) * (PW / CTX);

// dZ of four pixels: the gradients where the activations passed the ReLU
template <typename TA>
__device__ __forceinline__ float4 relu_grad4(const float* dA, const TA* act) {
    const float4 g = ldf4(dA, true), a = ldf4(act, true);
    return make_float4(a.x > 0.0f ? g.x : 0.0f, a.y > 0.0f ? g.y : 0.0f, a.z > 0.0f ? g.z : 0.0f, a.w > 0.0f ? g.w : 0.0f);
}

// Rows y0 - 1 .. y0 + ROWS - 2 and columns x0 - 1 .. x0 + COLS of a channel-major image's channels
// c0 .. c0 + N - 1, zeros outside the patch, to dst[c * CPITCH + row * RPITCH + column].  get4(g) and
// get1(g) read at index g of the image.
template <int N, int ROWS, int COLS, int CPITCH, int RPITCH, int NT, typename G4, typename G1>
__device__ __forceinline__ void load_halo(float* dst, size_t image, int y0, int x0, const G4& get4, const G1& get1) {
    constexpr int PARTS = COLS / 4;
    for (int q = threadIdx.x; q < N * ROWS * PARTS; q += NT) {
        const int part = q % PARTS, yy = (q / PARTS) % ROWS, c = q / (PARTS * ROWS);
        const int gy = y0 + yy - 1, gx = x0 + 4 * part;
        const bool in = gy >= 0 && gy < PH;
        const size_t g = image + static_cast<size_t>(c) * PHW + gy * PW + gx;
        float* d = dst + c * CPITCH + yy * RPITCH + 4 * part + 1;
        const float4 v = in ? get4(g) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        d[0] = v.x, d[1] = v.y, d[2] = v.z, d[3] = v.w;
        if (part == 0) d[-1] = in && gx > 0 ? get1(g - 1) : 0.0f;
        if (part == PARTS - 1) d[4] = in && gx + 4 < PW ? get1(g + 4) : 0.0f;
    }
}

template <int CI, int CO, int MODE, typename TIN, typename TA>
__global__ void __launch_bounds__(8 * CO) conv3x3_kernel(const void* __restrict__ in, const TA* __restrict__ act,
                                                         const TA* __restrict__ w, const TA* __restrict__ bias,
                                                         void* __restrict__ out) {
    constexpr int CK = CI < CCK ? CI : CCK, NT = 8 * CO, ROWS = CTY + 2;
    extern __shared__ __align__(16) float sm[];
    float* wsm = sm;                                   // CI * 9 * CO
    float* tile = sm + CI * 9 * CO;                    // CK * ROWS * CPX, column s is pixel s - 1
    const int b = blockIdx.x / kCTiles, tl = blockIdx.x % kCTiles;
    const int ty0 = (tl / (PW / CTX)) * CTY, tx0 = (tl % (PW / CTX)) * CTX;
    const int tid = threadIdx.x, o0 = (tid / 64) * 8, x0 = 4 * (tid % 8), y = 2 * ((tid % 64) / 8);
    for (int q = tid; q < CI * 9 * CO; q += NT) wsm[q] = ldf(w + q);
    float2 acc[2][4][4];                               // [row][pixel][channel pair]
#pragma unroll
    for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int j = 0; j < 8; ++j)
            acc[j / 4][j % 4][e] = MODE == 0 ? make_float2(ldf(bias + o0 + 2 * e), ldf(bias + o0 + 2 * e + 1)) : make_float2(0.0f, 0.0f);
    const bool wide = (reinterpret_cast<uintptr_t>(in) & 15) == 0;
    for (int c0 = 0; c0 < CI; c0 += CK) {
        __syncthreads();                               // the previous round's readers are done
        const size_t image = (static_cast<size_t>(b) * CI + c0) * PHW;
        if constexpr (MODE == 0) {
            const TIN* src = static_cast<const TIN*>(in);
            load_halo<CK, ROWS, CTX, ROWS * CPX, CPX, NT>(
                tile, image, ty0, tx0, [&](size_t g) { return ldf4(src + g, wide); }, [&](size_t g) { return ldf(src + g); });
        } else {
            const float* src = static_cast<const float*>(in);
            load_halo<CK, ROWS, CTX, ROWS * CPX, CPX, NT>(
                tile, image, ty0, tx0, [&](size_t g) { return relu_grad4(src + g, act + g); },
                [&](size_t g) { return ldf(act + g) > 0.0f ? src[g] : 0.0f; });
        }
        __syncthreads();
#pragma unroll 1
        for (int c = 0; c < CK; ++c) {
            float win[4][6];
#pragma unroll
            for (int dy = 0; dy < 4; ++dy) {
                const float* r = tile + (c * ROWS + y + dy) * CPX + x0;
                const float4 a = *reinterpret_cast<const float4*>(r);
                const float2 d = *reinterpret_cast<const float2*>(r + 4);
                win[dy][0] = a.x, win[dy][1] = a.y, win[dy][2] = a.z, win[dy][3] = a.w, win[dy][4] = d.x, win[dy][5] = d.y;
            }
            const float4* wc = reinterpret_cast<const float4*>(wsm + (c0 + c) * 9 * CO + o0);
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
                const float4 wa = wc[tap * (CO / 4)], wb = wc[tap * (CO / 4) + 1];
                const float2 ww[4] = {make_float2(wa.x, wa.y), make_float2(wa.z, wa.w), make_float2(wb.x, wb.y), make_float2(wb.z, wb.w)};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float t = win[j / 4 + tap / 3][j % 4 + tap % 3];
                    const float2 v = make_float2(t, t);
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[j / 4][j % 4][e] = __ffma2_rn(ww[e], v, acc[j / 4][j % 4][e]);
                }
            }
        }
    }
#pragma unroll
    for (int o = 0; o < 16; ++o) {
        const int row = o / 8, ch = o % 8;
        const size_t at = (static_cast<size_t>(b) * CO + o0 + ch) * PHW + (ty0 + y + row) * PW + tx0 + x0;
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[j] = (ch & 1) ? acc[row][j][ch / 2].y : acc[row][j][ch / 2].x;
            if (MODE == 0) v[j] = fmaxf(v[j], 0.0f);
        }
        if constexpr (MODE == 0 && sizeof(TA) == 2) {
            const __half2 h[2] = {__floats2half2_rn(v[0], v[1]), __floats2half2_rn(v[2], v[3])};
            *reinterpret_cast<uint2*>(static_cast<TA*>(out) + at) = *reinterpret_cast<const uint2*>(h);
        } else {
            *reinterpret_cast<float4*>(static_cast<float*>(out) + at) = make_float4(v[0], v[1], v[2], v[3]);
        }
    }
}

template <int CI, int CO>
size_t conv_smem() {
    return sizeof(float) * (CI * 9 * CO + (CI < CCK ? CI : CCK) * (CTY + 2) * CPX);
}

// ------------------------------------------------------------- weight gradient
// dW[o][c][tap] += sum_pixels dZ[o][p] A[c][p + tap],  db[o] += sum_pixels dZ[o][p],
// dZ = dA * (act > 0).  A CTA loops over 16 x 16 tiles; a thread owns one input channel, four output
// channels (two packed FP32x2 pairs) and rows of pixels of a tile, along which it slides the 3 x 3
// window (three new inputs and one 16-byte dZ read a pixel serve 18 packed operations).  The sums of
// a CTA's pixel groups are added in shared memory, one atomic per weight and CTA.
// What bounds it: the FP32 pipe.  256 patches, layers 3 / 2 / 1: 0.26 / 0.26 / 0.075 ms; 0.77 / 0.48 / 0.54 ms
// with a nine-value window and two dZ reads per 18 multiply-adds and an atomic per thread.
template <int CI, int CO>
struct WgPlan {
    static constexpr int UNITS = CI * CO / 4;                    // (channel, four outputs)
    static constexpr int NT = 256, G = NT / UNITS;               // pixel groups
    static constexpr int CP = TH * TH + 1;                       // channel pitch: lanes on 32 channels, 32 banks
    static constexpr int ZP = CO + 4;                            // pixel pitch of dZ [pixel][output]
    static constexpr int FLOATS = ((CI * CP + 3) / 4) * 4 + T * T * ZP;
    static_assert(NT % UNITS == 0 && G <= 64, "plan");
};

template <int CI, int CO, typename TIN, typename TA>
__global__ void __launch_bounds__(256) wgrad_kernel(const TIN* __restrict__ A, const float* __restrict__ dA,
                                                    const TA* __restrict__ act, float* __restrict__ dW,
                                                    float* __restrict__ db, int n_tiles) {
    using P = WgPlan<CI, CO>;
    constexpr int G = P::G, SEG = G <= T ? 1 : G / T, W = T / SEG;   // a group takes rows y = g % 16 (+ 16 ..), segments of W pixels
    extern __shared__ __align__(16) float sm[];
    float* at = sm;                                     // [CI][CP]
    float* dz = sm + ((CI * P::CP + 3) / 4) * 4;        // [T * T][ZP]
    const int tid = threadIdx.x, u = tid % P::UNITS, g = tid / P::UNITS;
    const int c = u % CI, o0 = 4 * (u / CI);
    float2 acc[9][2];
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) acc[tap][0] = acc[tap][1] = make_float2(0.0f, 0.0f);
    float accb = 0.0f;                                  // db of output tid % CO, pixels tid / CO ..
    const bool wide = (reinterpret_cast<uintptr_t>(A) & 15) == 0;
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int b = tile / kTiles, tl = tile % kTiles;
        const int ty0 = (tl / (PW / T)) * T, tx0 = (tl % (PW / T)) * T;
        __syncthreads();   // previous tile's readers are done
        load_halo<CI, TH, T, P::CP, TH, P::NT>(
            at, static_cast<size_t>(b) * CI * PHW, ty0, tx0, [&](size_t i) { return ldf4(A + i, wide); },
            [&](size_t i) { return ldf(A + i); });
        for (int q = tid; q < CO * T * T / 4; q += P::NT) {
            const int x4 = 4 * (q % (T / 4)), yy = (q / (T / 4)) % T, oo = q / (T * T / 4);
            const size_t i = (static_cast<size_t>(b) * CO + oo) * PHW + (ty0 + yy) * PW + tx0 + x4;
            const float4 v = relu_grad4(dA + i, act + i);
            float* d = dz + (yy * T + x4) * P::ZP + oo;
            d[0] = v.x, d[P::ZP] = v.y, d[2 * P::ZP] = v.z, d[3 * P::ZP] = v.w;
        }
        __syncthreads();
        for (int p = tid / CO; p < T * T; p += P::NT / CO) accb += dz[p * P::ZP + tid % CO];
        for (int y = g / SEG; y < T; y += G / SEG) {
            const int xs = (g % SEG) * W;
            const float* a = at + c * P::CP + y * TH + xs;
            const float* z = dz + (y * T + xs) * P::ZP + o0;
            float w0[3], w1[3];
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                w0[dy] = a[dy * TH];
                w1[dy] = a[dy * TH + 1];
            }
#pragma unroll
            for (int x = 0; x < W; ++x) {
                const float4 zz = *reinterpret_cast<const float4*>(z + x * P::ZP);
                const float2 za = make_float2(zz.x, zz.y), zb = make_float2(zz.z, zz.w);
#pragma unroll
                for (int dy = 0; dy < 3; ++dy) {
                    const float w2 = a[dy * TH + x + 2];
                    const float win[3] = {w0[dy], w1[dy], w2};
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        const float2 v = make_float2(win[dx], win[dx]);
                        acc[3 * dy + dx][0] = __ffma2_rn(za, v, acc[3 * dy + dx][0]);
                        acc[3 * dy + dx][1] = __ffma2_rn(zb, v, acc[3 * dy + dx][1]);
                    }
                    w0[dy] = w1[dy];
                    w1[dy] = w2;
                }
            }
        }
    }
    // the CTA's sums, weight by weight: shared-memory atomics over the pixel groups, then one global each
    __syncthreads();
    float* red = sm;                                    // [CO][CI][9], then db [CO]
    for (int q = tid; q < CO * CI * 9 + CO; q += P::NT) red[q] = 0.0f;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int tap = 0; tap < 9; ++tap)
            atomicAdd(&red[((o0 + j) * CI + c) * 9 + tap], (j & 1) ? acc[tap][j / 2].y : acc[tap][j / 2].x);
    atomicAdd(&red[CO * CI * 9 + tid % CO], accb);
    __syncthreads();
    for (int q = tid; q < CO * CI * 9; q += P::NT) atomicAdd(&dW[q], red[q]);
    if (tid < CO) atomicAdd(&db[tid], red[CO * CI * 9 + tid]);
}

template <int CI, int CO>
size_t wgrad_smem() {
    const int red = CO * CI * 9 + CO;
    return sizeof(float) * static_cast<size_t>(WgPlan<CI, CO>::FLOATS > red ? WgPlan<CI, CO>::FLOATS : red);
}

// ------------------------------------------------------------------- head
// logit = b4 + sum_c W4[c] A3[c][p].  Training: loss += BCE, dlogit = (sigmoid - m) / N,
// dA3[c][p] = W4[c] dlogit, dW4[c] += dlogit A3[c][p], db4 += dlogit.  Inference: prob.
template <typename TA>
__global__ void __launch_bounds__(256) head_kernel(const TA* __restrict__ A3, const uint8_t* __restrict__ mask,
                                                   const TA* __restrict__ pf16, int B, float inv_n,
                                                   float* __restrict__ dA3, float* __restrict__ grad,
                                                   float* __restrict__ loss, float* __restrict__ prob) {
    __shared__ float red[8][18];
    const int64_t q = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x;   // pixel over the batch
    float part[18];
#pragma unroll
    for (int j = 0; j < 18; ++j) part[j] = 0.0f;
    if (q < static_cast<int64_t>(B) * PHW) {
        const int64_t b = q / PHW, p = q % PHW;
        float a[16];
        float s = ldf(pf16 + OB4);
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            a[c] = ldf(A3 + (b * 16 + c) * PHW + p);
            s = fmaf(ldf(pf16 + OW4 + c), a[c], s);
        }
        const float pr = 1.0f / (1.0f + expf(-s));
        if (prob) prob[q] = pr;
        if (mask) {
            const float m = mask[q] ? 1.0f : 0.0f;
            part[17] = fmaxf(s, 0.0f) - s * m + log1pf(expf(-fabsf(s)));
            const float ds = (pr - m) * inv_n;
            part[16] = ds;
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                part[c] = ds * a[c];
                dA3[(b * 16 + c) * PHW + p] = ds * ldf(pf16 + OW4 + c);
            }
        }
    }
    if (!mask) return;
    // warp then block reduction of the 16 + 1 head gradients and the loss
#pragma unroll
    for (int j = 0; j < 18; ++j)
        for (int off = 16; off > 0; off >>= 1) part[j] += __shfl_xor_sync(0xffffffffu, part[j], off);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (lane == 0)
        for (int j = 0; j < 18; ++j) red[warp][j] = part[j];
    __syncthreads();
    if (threadIdx.x < 18) {
        float s = 0.0f;
        for (int w8 = 0; w8 < 8; ++w8) s += red[w8][threadIdx.x];
        if (threadIdx.x < 17)
            atomicAdd(&grad[OW4 + threadIdx.x], s);      // W4[0..15] then b4 (OB4 = OW4 + 16)
        else
            atomicAdd(loss, s);
    }
}

// ------------------------------------------------------- optimiser / weights
// TA copies of every parameter (rounded once from the FP32 masters) and the transposed /
// flipped layouts the convolutions read.
template <typename TA>
struct Wts {
    TA* pf16;                   // [NPAR] flat
    TA *wf1, *wf2, *wf3;        // forward  [CI][9][CO]
    TA *wb3, *wb2;              // backward [CO_fwd][9][CI_fwd], taps flipped
    unsigned char* pack;        // fp16: the tensor-core forward pass's operands (rfi_pack2, rfi_pack3)
};

template <typename TA>
__global__ void transform_kernel(const float* __restrict__ p, Wts<TA> w) {
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < NPAR; q += gridDim.x * blockDim.x) {
        TA h;
        stf(&h, p[q]);
        w.pf16[q] = h;
        int o, c, tap, ci, co;
        TA* fwd = nullptr;
        TA* bwd = nullptr;
        int off;
        if (q < OB1) {
            off = q - OW1; ci = 1; co = 16; fwd = w.wf1;
        } else if (q >= OW2 && q < OB2) {
            off = q - OW2; ci = 16; co = 32; fwd = w.wf2; bwd = w.wb2;
        } else if (q >= OW3 && q < OB3) {
            off = q - OW3; ci = 32; co = 16; fwd = w.wf3; bwd = w.wb3;
        } else {
            continue;
        }
        o = off / (ci * 9);
        c = (off / 9) % ci;
        tap = off % 9;
        fwd[(c * 9 + tap) * co + o] = h;                         // [c][tap][o]
        if constexpr (sizeof(TA) == 2) {
            if (ci > 1) *reinterpret_cast<TA*>(w.pack + (ci == 16 ? gbx::rfi_pack2(o, c, tap) : gbx::rfi_pack3(o, c, tap))) = h;
        }
        if (bwd) bwd[(o * 9 + (8 - tap)) * ci + c] = h;          // [o][8 - tap][c]
    }
}

// err: the network's error word; gradients of a forward pass whose wait ran out are not applied
__global__ void adam_kernel(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ g, float lr, float b1t, float b2t, const unsigned* __restrict__ err) {
    if (*err) return;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < NPAR; q += gridDim.x * blockDim.x) {
        const float gq = g[q];
        const float mq = b1 * m[q] + (1.0f - b1) * gq;
        const float vq = b2 * v[q] + (1.0f - b2) * gq * gq;
        m[q] = mq;
        v[q] = vq;
        p[q] -= lr * (mq / (1.0f - b1t)) / (sqrtf(vq / (1.0f - b2t)) + eps);
    }
}

// ------------------------------------------------------------ patch stats
// A warp takes a patch: its 4096 powers in registers (lane: two columns of each of the 64 rows), the
// two middle ranks of the powers and of the absolute deviations by bisection over the bit patterns
// of the floats between their extremes -- count the values at or below the middle one, until the
// bound falls between the two middle values (some 14 times; where they are equal 25 to 31) -- then
// the Eq. 4 flags and the compressed network input.  No shared memory, no barrier.
// What bounds it: dependent issue at 10 warps an SM (168 registers), half of it the counting, about 2
// instructions a value and step.  4096 patches: 0.145 ms (0.175 ms always bisecting to the last
// bit); 1.44 ms with two bitonic sorts of the patch in shared memory (78 barriers each).

// the floats in the order of their values as unsigned integers, and back
__device__ __forceinline__ uint32_t key_of(float f) {
    const uint32_t u = __float_as_uint(f);
    return u & 0x80000000u ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float of_key(uint32_t k) { return __uint_as_float(k & 0x80000000u ? k & 0x7fffffffu : ~k); }

// Mean of the two middle values of the warp's 4096 values get(q), q < 128 a lane (NaN sorts last).
template <typename Get>
__device__ __forceinline__ float median4096(const Get& get) {
    constexpr int kPer = PHW / 32;
    float mn = INFINITY, mx = -INFINITY;                   // (fminf and fmaxf pass NaN over)
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        mn = fminf(mn, get(q));
        mx = fmaxf(mx, get(q));
    }
    uint32_t lo = __reduce_min_sync(0xffffffffu, key_of(mn)), hi = __reduce_max_sync(0xffffffffu, key_of(mx));
    auto at_or_below = [&](float t) {
        int n = 0;
#pragma unroll
        for (int q = 0; q < kPer; ++q) n += get(q) <= t;
        return __reduce_add_sync(0xffffffffu, n);
    };
    // the smallest value with 2048 at or below it, or the first bound met with exactly 2048
    float t = 0.0f;
    int n = 0;
    while (lo < hi) {
        const uint32_t mid = lo + (hi - lo) / 2;
        t = of_key(mid);
        n = at_or_below(t);
        if (n == PHW / 2) break;
        if (n > PHW / 2) hi = mid;
        else lo = mid + 1;
    }
    if (n != PHW / 2) {
        t = of_key(lo);
        if (at_or_below(t) > PHW / 2) return 0.5f * (t + t);
    }
    float a = -INFINITY;                                   // the largest value at or below t
#pragma unroll
    for (int q = 0; q < kPer; ++q) a = get(q) <= t ? fmaxf(a, get(q)) : a;
    a = of_key(__reduce_max_sync(0xffffffffu, key_of(a)));
    float next = INFINITY;                                 // the next larger one
#pragma unroll
    for (int q = 0; q < kPer; ++q) next = get(q) > t ? fminf(next, get(q)) : next;
    return 0.5f * (a + of_key(__reduce_min_sync(0xffffffffu, key_of(next))));
}

__global__ void __launch_bounds__(128, 3) patch_kernel(const float* __restrict__ P, int B, int n_dump, int n_chan, float M,
                                                       __half* __restrict__ x, uint8_t* __restrict__ flags,
                                                       float* __restrict__ stats) {
    const int nkw = n_chan / PW, ndw = n_dump / PH, lane = threadIdx.x % 32;
    const int b = blockIdx.x * 4 + threadIdx.x / 32;
    if (b >= B) return;
    const int kw = b % nkw, dw = (b / nkw) % ndw, i = b / (nkw * ndw);
    const float* src = P + (static_cast<int64_t>(i) * n_dump + dw * PH) * n_chan + kw * PW + 2 * lane;
    const bool wide = !(reinterpret_cast<uintptr_t>(P) & 7);   // rows are multiples of 256 bytes: the base decides
    auto row = [&](int h) {
        const float* r = src + static_cast<int64_t>(h) * n_chan;
        return wide ? __ldg(reinterpret_cast<const float2*>(r)) : make_float2(__ldg(r), __ldg(r + 1));
    };
    float v[PHW / 32];
#pragma unroll
    for (int h = 0; h < PH; ++h) {
        const float2 t = row(h);
        v[2 * h] = t.x;
        v[2 * h + 1] = t.y;
    }
    const float med = median4096([&](int q) { return v[q]; });
    const float mad = median4096([&](int q) { return fabsf(v[q] - med); });
    const float sig = mad / 0.6745f, thr = M * sig;
    const bool pair = !((reinterpret_cast<uintptr_t>(x) & 3) | (reinterpret_cast<uintptr_t>(flags) & 1));
#pragma unroll 4
    for (int h = 0; h < PH; ++h) {                          // (read again: from the registers it would have to be unrolled)
        const int64_t o = static_cast<int64_t>(b) * PHW + h * PW + 2 * lane;
        const float2 t = row(h);
        float u[2];
        uint8_t f[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float dev = (e ? t.y : t.x) - med;
            f[e] = fabsf(dev) > thr ? 1 : 0;
            const float r = sig > 0.0f ? dev / sig : 0.0f;
            u[e] = x ? copysignf(log1pf(fabsf(r)), r) : 0.0f;
        }
        if (pair) {
            if (flags) *reinterpret_cast<uchar2*>(flags + o) = make_uchar2(f[0], f[1]);
            if (x) *reinterpret_cast<__half2*>(x + o) = __floats2half2_rn(u[0], u[1]);
        } else {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (flags) flags[o + e] = f[e];
                if (x) x[o + e] = __float2half_rn(u[e]);
            }
        }
    }
    if (stats && lane == 0) {
        stats[2 * b] = med;
        stats[2 * b + 1] = mad;
    }
}

}  // namespace

// ===================================================================== C ABI

struct rfi_net {
    int max_batch = 0;
    int step = 0;
    int fp32 = 0;                        // weights and activations in FP32 (rfi_create_fp32), else FP16
    float *p = nullptr, *m = nullptr, *v = nullptr, *g = nullptr, *loss = nullptr;
    void* w[7] = {};                     // Wts<TA>: pf16, wf1, wf2, wf3, wb3, wb2, pack
    unsigned* err = nullptr;             // device error word of the tensor-core kernel's bounded waits
    void *A1 = nullptr, *A2 = nullptr, *A3 = nullptr;   // TA activations
    float *dA1 = nullptr, *dA2 = nullptr, *dA3 = nullptr;
    int n_sm = 0;
};

namespace {

int rfail(int code, const char* what, cudaError_t e = cudaSuccess) {
    char buf[256];
    snprintf(buf, sizeof buf, "%s%s%s", what, e != cudaSuccess ? ": " : "", e != cudaSuccess ? cudaGetErrorString(e) : "");
    gbx::set_last_error(buf);
    return code;
}

#define RCU(call)                                                     \
    do {                                                              \
        cudaError_t e_ = (call);                                      \
        if (e_ != cudaSuccess) return rfail(CORR_E_CUDA, #call, e_);  \
    } while (0)

template <typename TA>
Wts<TA> wts(rfi_net* n) {
    Wts<TA> w;
    w.pf16 = static_cast<TA*>(n->w[0]);
    w.wf1 = static_cast<TA*>(n->w[1]);
    w.wf2 = static_cast<TA*>(n->w[2]);
    w.wf3 = static_cast<TA*>(n->w[3]);
    w.wb3 = static_cast<TA*>(n->w[4]);
    w.wb2 = static_cast<TA*>(n->w[5]);
    w.pack = static_cast<unsigned char*>(n->w[6]);
    return w;
}

template <int CI, int CO, int MODE, typename TIN, typename TA>
cudaError_t conv(const void* in, const TA* act, const TA* w, const TA* bias, void* out, int B, cudaStream_t s) {
    const size_t smem = conv_smem<CI, CO>();
    auto kern = conv3x3_kernel<CI, CO, MODE, TIN, TA>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    kern<<<B * kCTiles, 8 * CO, smem, s>>>(in, act, w, bias, out);
    return cudaGetLastError();
}

template <int CI, int CO, typename TIN, typename TA>
cudaError_t wgrad(const TIN* A, const float* dA, const TA* act, float* dW, float* db, int B, int n_sm,
                  cudaStream_t s) {
    const size_t smem = wgrad_smem<CI, CO>();
    auto kern = wgrad_kernel<CI, CO, TIN, TA>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    const int n_tiles = B * kTiles;
    const int grid = std::max(1, std::min(n_tiles, 3 * n_sm));
    kern<<<grid, 256, smem, s>>>(A, dA, act, dW, db, n_tiles);
    return cudaGetLastError();
}

template <typename TA>
int forward_t(rfi_net* n, const uint16_t* x, int B, cudaStream_t s) {
    const Wts<TA> w = wts<TA>(n);
    TA *A1 = static_cast<TA*>(n->A1), *A2 = static_cast<TA*>(n->A2), *A3 = static_cast<TA*>(n->A3);
    RCU((conv<1, 16, 0, __half, TA>(x, nullptr, w.wf1, w.pf16 + OB1, A1, B, s)));
    RCU((conv<16, 32, 0, TA, TA>(A1, nullptr, w.wf2, w.pf16 + OB2, A2, B, s)));
    RCU((conv<32, 16, 0, TA, TA>(A2, nullptr, w.wf3, w.pf16 + OB3, A3, B, s)));
    return CORR_OK;
}

// The FP16 flagger's forward pass on the tensor cores: probabilities and / or the activations a
// backward pass reads (keep)
int forward_tc(rfi_net* n, const uint16_t* x, int B, float* prob, bool keep, cudaStream_t s) {
    const Wts<__half> w = wts<__half>(n);
    gbx::RfiFwd f{};
    f.x = reinterpret_cast<const __half*>(x);
    f.pack = w.pack;
    f.w1 = w.pf16 + OW1;
    f.b1 = w.pf16 + OB1;
    f.b2 = w.pf16 + OB2;
    f.b3 = w.pf16 + OB3;
    f.w4 = w.pf16 + OW4;
    f.b4 = w.pf16 + OB4;
    f.prob = prob;
    if (keep) {
        f.A1 = static_cast<__half*>(n->A1);
        f.A2 = static_cast<__half*>(n->A2);
        f.A3 = static_cast<__half*>(n->A3);
    }
    f.B = B;
    f.err = n->err;
    RCU(gbx::launch_rfi_forward_tc(f, n->n_sm, s));
    return CORR_OK;
}

template <typename TA>
int forward_backward_t(rfi_net* n, const uint16_t* x, const uint8_t* mask, int B, cudaStream_t s) {
    RCU(cudaMemsetAsync(n->g, 0, sizeof(float) * NPAR, s));
    RCU(cudaMemsetAsync(n->loss, 0, sizeof(float), s));
    if constexpr (sizeof(TA) == 2) {
        // 16-byte loads of the patches: any other alignment takes the CUDA-core layers
        if (int rc = reinterpret_cast<uintptr_t>(x) & 15 ? forward_t<TA>(n, x, B, s) : forward_tc(n, x, B, nullptr, true, s)) return rc;
    } else {
        if (int rc = forward_t<TA>(n, x, B, s)) return rc;
    }
    const Wts<TA> w = wts<TA>(n);
    TA *A1 = static_cast<TA*>(n->A1), *A2 = static_cast<TA*>(n->A2), *A3 = static_cast<TA*>(n->A3);
    const int64_t npx = static_cast<int64_t>(B) * PHW;
    head_kernel<TA><<<static_cast<int>((npx + 255) / 256), 256, 0, s>>>(A3, mask, w.pf16, B, 1.0f / npx, n->dA3,
                                                                         n->g, n->loss, nullptr);
    RCU(cudaGetLastError());
    RCU((wgrad<32, 16, TA, TA>(A2, n->dA3, A3, n->g + OW3, n->g + OB3, B, n->n_sm, s)));
    RCU((conv<16, 32, 1, TA, TA>(n->dA3, A3, w.wb3, nullptr, n->dA2, B, s)));
    RCU((wgrad<16, 32, TA, TA>(A1, n->dA2, A2, n->g + OW2, n->g + OB2, B, n->n_sm, s)));
    RCU((conv<32, 16, 1, TA, TA>(n->dA2, A2, w.wb2, nullptr, n->dA1, B, s)));
    RCU((wgrad<1, 16, __half, TA>(reinterpret_cast<const __half*>(x), n->dA1, A1, n->g + OW1, n->g + OB1, B,
                                  n->n_sm, s)));
    return CORR_OK;
}

int forward_backward(rfi_net* n, const uint16_t* x, const uint8_t* mask, int B, cudaStream_t s) {
    return n->fp32 ? forward_backward_t<float>(n, x, mask, B, s) : forward_backward_t<__half>(n, x, mask, B, s);
}

int transform(rfi_net* n, cudaStream_t s) {
    if (n->fp32)
        transform_kernel<float><<<(NPAR + 255) / 256, 256, 0, s>>>(n->p, wts<float>(n));
    else
        transform_kernel<__half><<<(NPAR + 255) / 256, 256, 0, s>>>(n->p, wts<__half>(n));
    RCU(cudaGetLastError());
    return CORR_OK;
}

int head_infer(rfi_net* n, int B, float* prob, cudaStream_t s) {
    const int64_t npx = static_cast<int64_t>(B) * PHW;
    const int grid = static_cast<int>((npx + 255) / 256);
    if (n->fp32)
        head_kernel<float><<<grid, 256, 0, s>>>(static_cast<const float*>(n->A3), nullptr, wts<float>(n).pf16, B, 0.0f,
                                                nullptr, nullptr, nullptr, prob);
    else
        head_kernel<__half><<<grid, 256, 0, s>>>(static_cast<const __half*>(n->A3), nullptr, wts<__half>(n).pf16, B,
                                                 0.0f, nullptr, nullptr, nullptr, prob);
    RCU(cudaGetLastError());
    return CORR_OK;
}

// After a synchronisation: a bounded wait of the tensor-core kernel ran out since the last check
int check_err(rfi_net* n) {
    unsigned err = 0;
    RCU(cudaMemcpy(&err, n->err, sizeof err, cudaMemcpyDeviceToHost));
    if (!err) return CORR_OK;
    RCU(cudaMemset(n->err, 0, sizeof err));
    return rfail(CORR_E_TIMEOUT, "a kernel wait of the flagger timed out; results since the last synchronous call are invalid");
}

int check_batch(rfi_net* n, const void* x, int B) {
    if (!n) return rfail(CORR_E_INVAL, "null network");
    if (!x || B < 1 || B > n->max_batch) return rfail(CORR_E_INVAL, "batch must be 1..max_batch with inputs given");
    return CORR_OK;
}

int create(rfi_net_t** out, int max_batch, int fp32) {
    if (!out || max_batch < 1) return rfail(CORR_E_INVAL, "rfi_create: bad arguments");
    *out = nullptr;
    rfi_net* n = new rfi_net();
    n->max_batch = max_batch;
    n->fp32 = fp32;
    auto bail = [&](cudaError_t e) {
        rfi_destroy(n);
        return rfail(CORR_E_NOMEM, "rfi_create: allocation", e);
    };
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n->n_sm, cudaDevAttrMultiProcessorCount, dev);
    const size_t px = static_cast<size_t>(max_batch) * PHW;
    const size_t ta = fp32 ? sizeof(float) : sizeof(__half);
    void** f32[] = {reinterpret_cast<void**>(&n->p), reinterpret_cast<void**>(&n->m), reinterpret_cast<void**>(&n->v),
                    reinterpret_cast<void**>(&n->g)};
    for (void** q : f32)
        if (e == cudaSuccess) e = cudaMalloc(q, sizeof(float) * NPAR);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->loss), sizeof(float));
    const size_t wn[6] = {NPAR, 144, 4608, 4608, 4608, 4608};
    for (int q = 0; q < 6; ++q)
        if (e == cudaSuccess) e = cudaMalloc(&n->w[q], ta * wn[q]);
    if (e == cudaSuccess) e = cudaMalloc(&n->w[6], gbx::kRfiPackBytes);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->err), sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemset(n->err, 0, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMalloc(&n->A1, ta * px * 16);
    if (e == cudaSuccess) e = cudaMalloc(&n->A2, ta * px * 32);
    if (e == cudaSuccess) e = cudaMalloc(&n->A3, ta * px * 16);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->dA1), sizeof(float) * px * 16);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->dA2), sizeof(float) * px * 32);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&n->dA3), sizeof(float) * px * 16);
    if (e != cudaSuccess) return bail(e);
    for (void** q : f32)
        if ((e = cudaMemset(*q, 0, sizeof(float) * NPAR)) != cudaSuccess) return bail(e);
    if (transform(n, nullptr) != CORR_OK || cudaDeviceSynchronize() != cudaSuccess)
        return bail(cudaGetLastError());
    *out = n;
    return CORR_OK;
}

}  // namespace

extern "C" {

int rfi_n_params(void) { return NPAR; }

int rfi_create(rfi_net_t** out, int max_batch) { return create(out, max_batch, 0); }

int rfi_create_fp32(rfi_net_t** out, int max_batch) { return create(out, max_batch, 1); }

int rfi_destroy(rfi_net_t* n) {
    if (!n) return CORR_OK;
    void* bufs[] = {n->p, n->m, n->v, n->g, n->loss, n->w[0], n->w[1], n->w[2], n->w[3], n->w[4],
                    n->w[5], n->w[6], n->err, n->A1, n->A2, n->A3, n->dA1, n->dA2, n->dA3};
    for (void* b : bufs)
        if (b) cudaFree(b);
    delete n;
    return CORR_OK;
}

int rfi_set_params(rfi_net_t* n, const float* params) {
    if (!n || !params) return rfail(CORR_E_INVAL, "rfi_set_params: null argument");
    for (int q = 0; q < NPAR; ++q)
        if (!std::isfinite(params[q])) return rfail(CORR_E_INVAL, "rfi_set_params: non-finite parameter");
    RCU(cudaMemcpy(n->p, params, sizeof(float) * NPAR, cudaMemcpyHostToDevice));
    RCU(cudaMemset(n->m, 0, sizeof(float) * NPAR));
    RCU(cudaMemset(n->v, 0, sizeof(float) * NPAR));
    n->step = 0;
    if (int rc = transform(n, nullptr)) return rc;
    RCU(cudaDeviceSynchronize());
    return CORR_OK;
}

int rfi_get_params(rfi_net_t* n, float* params) {
    if (!n || !params) return rfail(CORR_E_INVAL, "rfi_get_params: null argument");
    RCU(cudaDeviceSynchronize());
    RCU(cudaMemcpy(params, n->p, sizeof(float) * NPAR, cudaMemcpyDeviceToHost));
    return check_err(n);
}

int rfi_loss_grad(rfi_net_t* n, const uint16_t* x, const uint8_t* mask, int B, float* loss, float* grad,
                  void* stream) {
    if (int rc = check_batch(n, x, B)) return rc;
    if (!mask || !loss) return rfail(CORR_E_INVAL, "rfi_loss_grad: mask and loss are required");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (int rc = forward_backward(n, x, mask, B, s)) return rc;
    RCU(cudaStreamSynchronize(s));
    RCU(cudaMemcpy(loss, n->loss, sizeof(float), cudaMemcpyDeviceToHost));
    *loss /= static_cast<float>(static_cast<int64_t>(B) * PHW);
    if (grad) RCU(cudaMemcpy(grad, n->g, sizeof(float) * NPAR, cudaMemcpyDeviceToHost));
    return check_err(n);
}

int rfi_train_step(rfi_net_t* n, const uint16_t* x, const uint8_t* mask, int B, float lr, float* loss,
                   void* stream) {
    if (int rc = check_batch(n, x, B)) return rc;
    if (!mask || !(lr > 0.0f)) return rfail(CORR_E_INVAL, "rfi_train_step: mask required and lr > 0");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (int rc = forward_backward(n, x, mask, B, s)) return rc;
    n->step += 1;
    const float b1t = std::pow(0.9f, static_cast<float>(n->step)), b2t = std::pow(0.999f, static_cast<float>(n->step));
    adam_kernel<<<(NPAR + 255) / 256, 256, 0, s>>>(n->p, n->m, n->v, n->g, lr, b1t, b2t, n->err);
    RCU(cudaGetLastError());
    if (int rc = transform(n, s)) return rc;
    if (loss) {
        RCU(cudaStreamSynchronize(s));
        RCU(cudaMemcpy(loss, n->loss, sizeof(float), cudaMemcpyDeviceToHost));
        *loss /= static_cast<float>(static_cast<int64_t>(B) * PHW);
        return check_err(n);
    }
    return CORR_OK;
}

int rfi_infer(rfi_net_t* n, const uint16_t* x, int B, float* prob, void* stream) {
    if (int rc = check_batch(n, x, B)) return rc;
    if (!prob) return rfail(CORR_E_INVAL, "rfi_infer: prob is null");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!n->fp32 && !(reinterpret_cast<uintptr_t>(x) & 15)) return forward_tc(n, x, B, prob, false, s);
    if (int rc = n->fp32 ? forward_t<float>(n, x, B, s) : forward_t<__half>(n, x, B, s)) return rc;
    return head_infer(n, B, prob, s);
}

int rfi_status(rfi_net_t* n, void* stream) {
    if (!n) return rfail(CORR_E_INVAL, "null network");
    RCU(cudaStreamSynchronize(static_cast<cudaStream_t>(stream)));
    return check_err(n);
}

int rfi_wait_selftest(rfi_net_t* n) {
    if (!n) return rfail(CORR_E_INVAL, "null network");
    RCU(gbx::launch_wait_selftest(n->err, nullptr, nullptr));
    RCU(cudaDeviceSynchronize());
    unsigned err = 0;
    RCU(cudaMemcpy(&err, n->err, sizeof err, cudaMemcpyDeviceToHost));
    return (err & gbx::ERR_WAIT_STAGE) ? CORR_OK : rfail(CORR_E_STATE, "the wait did not give up");
}

int rfi_patches(const float* power, int n_in, int n_dump, int n_chan, float M, uint16_t* x, uint8_t* mad_flags,
                float* stats, void* stream) {
    if (!power || n_in < 1 || n_dump < PH || n_chan < PW || n_dump % PH || n_chan % PW || !(M > 0.0f))
        return rfail(CORR_E_INVAL, "rfi_patches: need n_dump, n_chan multiples of 64 and M > 0");
    const int B = n_in * (n_dump / PH) * (n_chan / PW);
    patch_kernel<<<(B + 3) / 4, 128, 0, static_cast<cudaStream_t>(stream)>>>(power, B, n_dump, n_chan, M,
                                                                             reinterpret_cast<__half*>(x), mad_flags, stats);
    RCU(cudaGetLastError());
    return CORR_OK;
}

}  // extern "C"
