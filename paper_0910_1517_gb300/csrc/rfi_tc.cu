// rfi_tc.cu -- the learned flagger's forward pass (three 3x3 convolutions 1 -> 16 -> 32 -> 16, a 1x1
// convolution and the sigmoid) in one kernel, activations in shared memory, the two large layers on
// the tcgen05 tensor cores.
//
// A CTA takes strips of 8 output rows of a 64 x 64 patch.  Activations lie in shared memory as
// planes of 8 channels, one 16-byte piece per position; positions are numbered row by row with a
// pitch of 65, one column of zeros serving as the right edge of a row and the left edge of the next.
// A plane is then a no-swizzle K-major operand (core matrices of 8 positions x 8 channels), 128
// consecutive positions are the rows of one 128 x N x 16 MMA, and a tap (dy, dx) is the same
// operand 65 dy + dx - 1 positions on: the convolution is nine accumulating MMAs per 16 input
// channels with no im2col copy.  Halo rows are recomputed (12 rows of layer 1, 10 of layer 2 per 8
// rows of output).  Layer 1 (one input channel) runs on the CUDA cores, two channels a packed FP32x2
// operation.
//
// Rounding.  The tensor core adds the products of an output in another order than the CUDA-core
// kernels; where the FP32 sum lies next to a rounding boundary of fp16 the activation could round
// the other way, a whole fp16 step.  Activations near a boundary are therefore listed and summed
// again in FP32 in the CUDA-core order, one a thread.  How near is set by what the sums' errors follow:
// in layer 2, whose flips spread over nine positions and sixteen channels, the size of the terms
// (kTie2 x the mean of the output's |weights| x the sum of its 144 inputs; small sums of large
// terms are the ones that flip furthest from a boundary), in layer 3 32 FP32 steps of the sum.
// Largest differences of the probabilities from the CUDA-core order's, 40 x 4096 patches with as many
// networks: 3e-4 (median of the 40), 6.6e-4 (worst), relative 2-norm at most 6e-7; the same with
// twice and six times the margin.  With 64 steps of the sum in both layers, as fast within 10 %, 6e-4 and
// 1.2e-3; with 256, a third slower, 4e-4 and 8.7e-4.
// Against 64 bits neither order is further off: over ten networks x 512 patches each of random, large-bias,
// heavy-tailed, all-positive and trained weights the rms errors of the probabilities agree to 2e-4 (9.7e-6
// to 1.1e-4, the fp16 weights and activations), against 64-bit sums of fp16 activations to 2 %, and the
// gradients' to 3 %, either way.
//
// Roles: warp 8 issues the MMAs of a layer tile by tile (a commit each), warps 0-7 take the tiles as
// they complete: bias, ReLU, rounding to fp16, zeros outside the image, and the next layer's
// planes.  Two CTAs an SM overlap one's epilogues with the other's MMAs.  All waits are bounded.
//
// What bounds it: an MMA with N = 16 or 32 takes the tensor core about 40 cycles whatever its N, 144
// of them a strip (0.6 ms for 4096 patches), and the near ties' sums, one after another by
// definition, which little runs beside.  4096 patches, four launches: 1.9 ms; 10.95 ms with a CUDA-core kernel a
// layer and the head's (conv2 5.0, conv3 5.5, conv1 0.29, head 0.15 ms).  Layer 1's four positions a
// thread: with one, its weight loads took the pass to 1.97 ms.
#include <type_traits>

#include "common.cuh"
#include "rfi_tc.cuh"

namespace gbx {
namespace {

constexpr int kPatch = 64, kRows = 8, kPitch = 65;
constexpr int kStrips = kPatch / kRows;
constexpr int kRows1 = 12, kTiles2 = (10 * kPitch + 127) / 128, kTiles3 = (8 * kPitch + 127) / 128;
constexpr int kXPitch = 66;
constexpr int kPos1 = 912;                                // positions of an A1 plane (index position + 1)
constexpr int kPos2 = kTiles2 * 128 + 16;                 // ... of an A2 plane
static_assert(kTiles2 * 128 + 2 * kPitch + 2 <= kPos1 && kTiles3 * 128 + 2 * kPitch + 2 <= kPos2, "a tile reads within its planes");
constexpr int kEpiWarps = 8;
constexpr int kThreadsTc = (kEpiWarps + 1) * 32;

// near ties a layer of a strip can list.  With more of them (patches of one repeated value: a channel's
// positions are all near ties or none) the whole layer of the strip is summed in order instead: which
// of them found a place on the list would depend on the warps' timing.
constexpr int kMaxTies = 2048;
constexpr int kPosA3 = kTiles3 * 128;                     // A3 [8 channel pairs][position], where A1 was

struct Smem {
    static constexpr int pack = 0;
    static constexpr int A1 = pack + (kRfiPackBytes + 127) / 128 * 128;      // 2 planes
    static constexpr int A2 = A1 + 2 * kPos1 * 16;                           // 4 planes
    static constexpr int x = A2 + 4 * kPos2 * 16;                            // 14 input rows, FP32
    static constexpr int ties = x + 14 * kXPitch * 4;                        // list of near ties (position * 32 + channel)
    static constexpr int sum1 = ties + kMaxTies * 2;                         // layer 1's activations summed over channels, FP32
    static constexpr int total = sum1 + kPos1 * 4;
};
static_assert(8 * kPosA3 * 4 <= 2 * kPos1 * 16 && kTiles2 * 128 * 32 <= 65536, "A3 where A1 was; 16-bit list entries");
static_assert(Smem::total <= 112 * 1024, "two CTAs an SM");

struct alignas(16) Ctl {
    uint64_t done[kTiles2 + kTiles3];                     // a tile's MMAs are complete
    uint64_t wbar;                                        // weights landed
    uint32_t taddr;
    int fail, n_tie[2];                                   // near ties of layers 2 and 3
    float bias[16 + 32 + 16 + 16 + 1];                    // b1, b2, b3, w4, b4
    float4 w1[2][9][2];                                   // layer 1, [8 channels][tap][4 channels]
    float tie2[32];                                       // layer 2: kTie2 x the mean of an output's |weights|
};

// Near ties of layer 2: r > 0 within e of the middle between two fp16 numbers, where rounding turns;
// kTie2Cap r, a quarter to half of the way between the two, is the most it reaches (small sums of
// large terms would all be listed, and their flips weigh little).
constexpr float kTie2 = 8.0f / 16777216.0f, kTie2Cap = 1.0f / 8192.0f;
__device__ __forceinline__ bool near_tie2(float r, float e) {
    const float mid = __uint_as_float((__float_as_uint(r) & ~0x1fffu) | 0x1000u);
    return fabsf(r - mid) < fminf(e, r * kTie2Cap);
}

// ... of layer 3: r >= 0 within kTie3 FP32 steps of it: the 13 bits that fp16 drops lie around 0x1000
// (below fp16's normal numbers and above its largest the answer does not matter)
constexpr uint32_t kTie3 = 32;
__device__ __forceinline__ bool near_tie3(float r) {
    return ((__float_as_uint(r) - (0x1000u - kTie3)) & 0x1fffu) <= 2 * kTie3;
}

// A pair of activations (channels o and o + 1) from their sums without bias; their near ties, as the
// functions t0 and t1 find them, in mask
template <typename T0, typename T1>
__device__ __forceinline__ uint32_t round_pair(uint32_t v0, uint32_t v1, float b0, float b1, int o, uint32_t& mask, const T0& t0,
                                               const T1& t1) {
    const float r0 = fmaxf(__uint_as_float(v0) + b0, 0.0f), r1 = fmaxf(__uint_as_float(v1) + b1, 0.0f);
    const __half2 a = __floats2half2_rn(r0, r1);
    if (t0(r0)) mask |= 1u << o;
    if (t1(r1)) mask |= 2u << o;
    return *reinterpret_cast<const uint32_t*>(&a);
}

// w a + acc in FP32, rounded once, w and a fp16: the same value as of the operands converted first, in
// one instruction instead of three (flagging 4096 patches 2.05 -> 1.87 ms)
__device__ __forceinline__ float fma_half(unsigned short w, unsigned short a, float acc) {
    asm("fma.rn.f32.f16 %0, %1, %2, %0;" : "+f"(acc) : "h"(w), "h"(a));
    return acc;
}

// The activation of output channel o at plane index `at` (the tap (0, 0) of its position), summed in
// FP32 in the order of the CUDA-core kernels: bias, then channel by channel, tap by tap.  GROUPS
// planes of 8 channels of `pos` positions; wt: packed weights of (o, channel 0, tap 0), `wg` bytes
// from one group of 8 channels to the next, 1024 from tap to tap.
template <int GROUPS>
__device__ __forceinline__ __half sum_in_order(const unsigned char* planes, int pos, int at, const unsigned char* wt, int wg,
                                               float bias) {
    float acc = bias;
#pragma unroll 1
    for (int g = 0; g < GROUPS; ++g) {
        uint4 a[9], w[9];
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
            a[tap] = *reinterpret_cast<const uint4*>(planes + (g * pos + at + (tap / 3) * kPitch + tap % 3) * 16);
            w[tap] = *reinterpret_cast<const uint4*>(wt + g * wg + tap * 1024);
        }
#pragma unroll
        for (int ch = 0; ch < 8; ++ch)
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
                const uint32_t aw = (&a[tap].x)[ch / 2], ww = (&w[tap].x)[ch / 2];
                acc = fma_half(static_cast<unsigned short>(ww >> (16 * (ch & 1))), static_cast<unsigned short>(aw >> (16 * (ch & 1))), acc);
            }
    }
    return __float2half_rn(fmaxf(acc, 0.0f));
}

template <bool KEEP>
__global__ void __launch_bounds__(kThreadsTc, 2) rfi_forward_kernel(const RfiFwd p) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) Ctl c;
    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x) / 32, 0), lane = threadIdx.x % 32;
    const int tid = threadIdx.x;
    if (tid == 0) {
        for (uint64_t& b : c.done) mbar_init(&b, 1);
        mbar_init(&c.wbar, 1);
        fence_mbar_init();
        c.fail = 0;
        mbar_arrive_expect_tx(&c.wbar, kRfiPackBytes);
        bulk_g2s(smem + Smem::pack, p.pack, kRfiPackBytes, &c.wbar);
    }
    if (warp == kEpiWarps) {
        tmem_alloc(&c.taddr, 256);
        tmem_relinquish();
    }
    if (tid < 144) reinterpret_cast<float*>(c.w1)[((tid / 72) * 9 + tid % 9) * 8 + (tid / 9) % 8] = __half2float(p.w1[tid]);
    for (int q = tid; q < 81; q += kThreadsTc)
        c.bias[q] = __half2float(q < 16 ? p.b1[q] : q < 48 ? p.b2[q - 16] : q < 64 ? p.b3[q - 48] : q < 80 ? p.w4[q - 64] : p.b4[0]);
    // zero everything once: the guard positions before and after the planes.  (A3 overwrites A1's; only
    // positions outside the strip read them, whose sums are not used.)
    for (int q = tid; q < (Smem::total - Smem::A1) / 16; q += kThreadsTc)
        reinterpret_cast<uint4*>(smem + Smem::A1)[q] = make_uint4(0u, 0u, 0u, 0u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = __shfl_sync(0xffffffffu, c.taddr, 0);
    const uint32_t s0 = __shfl_sync(0xffffffffu, smem_u32(smem), 0);
    float* xs = reinterpret_cast<float*>(smem + Smem::x);
    float* sum1 = reinterpret_cast<float*>(smem + Smem::sum1);
    bool ok = mbar_wait_warp(&c.wbar, 0, p.err, ERR_WAIT_STAGE);
    if (tid < 32) {
        float m = 0.0f;
        for (int q = 0; q < 144; ++q)
            m += fabsf(__half2float(*reinterpret_cast<const __half*>(smem + Smem::pack + rfi_pack2(tid, q / 9, q % 9))));
        c.tie2[tid] = m * (kTie2 / 144.0f);
    }

    // this thread's 16 bytes of the strip's 14 input rows (y0 - 3 .. y0 + 10), zero outside the patch
    const int n_items = p.B * kStrips;
    auto load_x = [&](int it) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        const int gy = (it % kStrips) * kRows - 3 + tid / 8;
        if (it < n_items && tid < 14 * 8 && gy >= 0 && gy < kPatch)
            v = __ldg(reinterpret_cast<const uint4*>(p.x + (static_cast<int64_t>(it / kStrips) * kPatch + gy) * kPatch) + tid % 8);
        return v;
    };
    uint4 xv = load_x(blockIdx.x);
    uint32_t par = 0;
    // a layer's MMAs by the issuing warp, tile t's completion on done[base + t]; KG groups of 16
    // input channels (two planes each)
    auto issue = [&](auto kg_, int tiles, uint32_t a0, uint32_t pos, uint32_t b0, int N, int base) {
        constexpr int KG = decltype(kg_)::value;
        if (elect_one()) {
            const uint32_t idesc = idesc_f16_f32(128, N);
#pragma unroll 1
            for (int t = 0; t < tiles; ++t) {
                uint64_t da = smem_desc_noswizzle(a0 + t * 2048, pos * 16, 128);
                uint64_t db = smem_desc_noswizzle(b0, N * 16, 128);
#pragma unroll 1
                for (int dy = 0; dy < 3; ++dy) {
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                        for (int kg = 0; kg < KG; ++kg)
                            umma_f16(tm + t * N, da + dx + kg * 2 * pos, db + dx * 64 + kg * 2 * N, idesc,
                                     (dy | dx | kg) ? 1u : 0u);
                    da += kPitch;
                    db += 3 * 64;
                }
                umma_commit(&c.done[base + t]);
            }
        }
        __syncwarp();
    };
    unsigned short* ties = reinterpret_cast<unsigned short*>(smem + Smem::ties);
    // list channels `mask` of position q as near ties of layer 2 (which = 0) or 3
    auto list = [&](uint32_t mask, int q, int which) {
        if (!mask) return;
        for (int i = atomicAdd(&c.n_tie[which], __popc(mask)); mask; mask &= mask - 1, ++i)
            if (i < kMaxTies) ties[i] = static_cast<unsigned short>(q * 32 + __ffs(mask) - 1);
    };
    // n channels of pixel (gy, gx), pairs h, to the planar activations A [B][C][64][64]
    auto keep = [&](__half* A, int C, int n, const uint32_t* h, int64_t patch, int gy, int gx) {
        __half* o = A + (patch * C * kPatch + gy) * kPatch + gx;
#pragma unroll
        for (int e = 0; e < 32; ++e)
            if (e < n) o[e * kPatch * kPatch] = __ushort_as_half(static_cast<unsigned short>(h[e / 2] >> (16 * (e & 1))));
    };
    for (int it = blockIdx.x; it < n_items; it += gridDim.x, par ^= 1u) {
        const int64_t patch = it / kStrips;
        const int y0 = (it % kStrips) * kRows;
        if (tid < 2) c.n_tie[tid] = 0;
        if (tid < 14 * 8) {                                // columns 1 .. 64 of the row (0 and 65 stay zero)
            const uint32_t w[4] = {xv.x, xv.y, xv.z, xv.w};
            float* d = xs + (tid / 8) * kXPitch + 1 + (tid % 8) * 8;
#pragma unroll
            for (int e = 0; e < 8; ++e) d[e] = __half2float(__ushort_as_half(static_cast<unsigned short>(w[e / 2] >> (16 * (e & 1)))));
        }
        __syncthreads();
        xv = load_x(it + gridDim.x);
        // ---- layer 1: four positions (row r, column cc - 1) a thread, 8 channels at a time, channel pairs
        // in packed FP32x2, tap by tap: two 16-byte weight loads serve 16 packed operations
        if (warp < kEpiWarps) {
            int at[4];
            bool in[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int q = tid + j * kEpiWarps * 32, r = q / kPitch, cc = q % kPitch, gy = y0 - 2 + r;
                in[j] = cc > 0 && q < kRows1 * kPitch && gy >= 0 && gy < kPatch;
                at[j] = in[j] ? r * kXPitch + cc - 1 : 0;
            }
            float sum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
            for (int g = 0; g < 2; ++g) {
                float2 acc[4][4];
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[j][e] = make_float2(c.bias[8 * g + 2 * e], c.bias[8 * g + 2 * e + 1]);
#pragma unroll
                for (int tap = 0; tap < 9; ++tap) {
                    const float4 wa = c.w1[g][tap][0], wb = c.w1[g][tap][1];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float v = xs[at[j] + (tap / 3) * kXPitch + tap % 3];
                        const float2 vv = make_float2(v, v);
                        acc[j][0] = __ffma2_rn(make_float2(wa.x, wa.y), vv, acc[j][0]);
                        acc[j][1] = __ffma2_rn(make_float2(wa.z, wa.w), vv, acc[j][1]);
                        acc[j][2] = __ffma2_rn(make_float2(wb.x, wb.y), vv, acc[j][2]);
                        acc[j][3] = __ffma2_rn(make_float2(wb.z, wb.w), vv, acc[j][3]);
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int q = tid + j * kEpiWarps * 32;
                    uint32_t h[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float ax = fmaxf(acc[j][e].x, 0.0f), ay = fmaxf(acc[j][e].y, 0.0f);
                        const __half2 a = __floats2half2_rn(ax, ay);
                        h[e] = in[j] ? *reinterpret_cast<const uint32_t*>(&a) : 0u;
                        sum[j] += ax + ay;
                    }
                    if (q <= kRows1 * kPitch)              // (the position after the last row: its right edge)
                        reinterpret_cast<uint4*>(smem + Smem::A1)[g * kPos1 + q + 1] = make_uint4(h[0], h[1], h[2], h[3]);
                    const int r = q / kPitch;
                    if (g && q <= kRows1 * kPitch) sum1[q + 1] = in[j] ? sum[j] : 0.0f;
                    if (KEEP && in[j] && r >= 2 && r < 10) keep(p.A1 + g * 8 * kPatch * kPatch, 16, 8, h, patch, y0 - 2 + r, q % kPitch - 1);
                }
            }
            fence_proxy_async_smem();
        }
        __syncthreads();
        // ---- layer 2
        if (warp == kEpiWarps) {
            tc_fence_after();
            issue(std::integral_constant<int, 1>{}, kTiles2, s0 + Smem::A1, kPos1, s0 + Smem::pack, 32, 0);
        } else {
            const int q4 = warp & 3, half = warp >> 2;
            for (int t = half; t < kTiles2; t += 2) {
                ok = ok && mbar_wait_warp(&c.done[t], par, p.err, ERR_WAIT_MMA);
                tc_fence_after();
                uint32_t v[32];
                tmem_ld32(tm + (static_cast<uint32_t>(32 * q4) << 16) + t * 32, v);
                tmem_wait_ld();
                const int q = t * 128 + 32 * q4 + lane, r = q / kPitch, cc = q % kPitch, gy = y0 - 1 + r;
                const bool in = cc > 0 && r < 10 && gy >= 0 && gy < kPatch;
                float near = 0.0f;                         // the inputs' sum over channels and taps
#pragma unroll
                for (int tap = 0; tap < 9; ++tap) near += sum1[q + (tap / 3) * kPitch + tap % 3];
                uint32_t h[16], mask = 0;
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    h[e] = round_pair(
                        v[2 * e], v[2 * e + 1], c.bias[16 + 2 * e], c.bias[17 + 2 * e], 2 * e, mask,
                        [&](float r) { return near_tie2(r, near * c.tie2[2 * e]); },
                        [&](float r) { return near_tie2(r, near * c.tie2[2 * e + 1]); });
                    if (!in) h[e] = 0u;
                }
                uint4* d = reinterpret_cast<uint4*>(smem + Smem::A2) + q + 1;
#pragma unroll
                for (int g = 0; g < 4; ++g) d[g * kPos2] = make_uint4(h[4 * g], h[4 * g + 1], h[4 * g + 2], h[4 * g + 3]);
                list(in ? mask : 0u, q, 0);
            }
            tc_fence_before();
        }
        __syncthreads();
        const int ties2 = c.n_tie[0];
        for (int i = tid; i < (ties2 > kMaxTies ? 10 * kPatch * 32 : ties2); i += kThreadsTc) {
            int q, o;
            if (ties2 <= kMaxTies) {
                q = ties[i] >> 5, o = ties[i] & 31;
            } else {                                       // every position inside the image, channel by channel
                const int r = (i / kPatch) % 10;
                if (y0 - 1 + r < 0 || y0 - 1 + r >= kPatch) continue;
                q = r * kPitch + i % kPatch + 1, o = i / (10 * kPatch);
            }
            reinterpret_cast<__half*>(smem + Smem::A2)[((o / 8) * kPos2 + q + 1) * 8 + o % 8] =
                sum_in_order<2>(smem + Smem::A1, kPos1, q, smem + Smem::pack + rfi_pack2(o, 0, 0), 512, c.bias[16 + o]);
        }
        fence_proxy_async_smem();
        __syncthreads();
        if (KEEP)                                          // (read back once repaired)
            for (int i = tid; i < kRows * kPatch; i += kThreadsTc) {
                const int r = i / kPatch + 1, gx = i % kPatch;
                uint32_t h[16];
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const uint4 u = reinterpret_cast<const uint4*>(smem + Smem::A2)[g * kPos2 + r * kPitch + gx + 2];
                    h[4 * g] = u.x, h[4 * g + 1] = u.y, h[4 * g + 2] = u.z, h[4 * g + 3] = u.w;
                }
                keep(p.A2, 32, 32, h, patch, y0 - 1 + r, gx);
            }
        // ---- layer 3
        uint32_t* a3 = reinterpret_cast<uint32_t*>(smem + Smem::A1);
        if (warp == kEpiWarps) {
            tc_fence_after();
            issue(std::integral_constant<int, 2>{}, kTiles3, s0 + Smem::A2, kPos2, s0 + Smem::pack + kRfiW2Bytes, 16, kTiles2);
        } else {
            const int q4 = warp & 3, half = warp >> 2;
            for (int t = half; t < kTiles3; t += 2) {
                ok = ok && mbar_wait_warp(&c.done[kTiles2 + t], par, p.err, ERR_WAIT_MMA);
                tc_fence_after();
                uint32_t v[16];
                tmem_ld16(tm + (static_cast<uint32_t>(32 * q4) << 16) + t * 16, v);
                tmem_wait_ld();
                const int q = t * 128 + 32 * q4 + lane, r = q / kPitch, cc = q % kPitch;
                uint32_t mask = 0;
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    a3[e * kPosA3 + q] =
                        round_pair(v[2 * e], v[2 * e + 1], c.bias[48 + 2 * e], c.bias[49 + 2 * e], 2 * e, mask, near_tie3, near_tie3);
                list(cc > 0 && r < kRows ? mask : 0u, q, 1);
            }
            tc_fence_before();
            if (!ok) *(volatile int*)&c.fail = 1;
        }
        __syncthreads();
        const int ties3 = c.n_tie[1];
        for (int i = tid; i < (ties3 > kMaxTies ? kRows * kPatch * 16 : ties3); i += kThreadsTc) {
            const bool all = ties3 > kMaxTies;
            const int q = all ? (i / kPatch) % kRows * kPitch + i % kPatch + 1 : ties[i] >> 5;
            const int o = all ? i / (kRows * kPatch) : ties[i] & 31;
            reinterpret_cast<__half*>(a3)[((o / 2) * kPosA3 + q) * 2 + (o & 1)] =
                sum_in_order<4>(smem + Smem::A2, kPos2, q, smem + Smem::pack + rfi_pack3(o, 0, 0), 256, c.bias[48 + o]);
        }
        __syncthreads();
        // ---- head: the 1x1 convolution and the sigmoid
        for (int i = tid; i < kRows * kPatch; i += kThreadsTc) {
            const int gy = y0 + i / kPatch, gx = i % kPatch, q = (i / kPatch) * kPitch + gx + 1;
            uint32_t h[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) h[e] = a3[e * kPosA3 + q];
            if (KEEP) keep(p.A3, 16, 16, h, patch, gy, gx);
            if (p.prob) {
                float s = c.bias[80];
#pragma unroll
                for (int e = 0; e < 16; ++e)
                    s = fmaf(c.bias[64 + e], __half2float(__ushort_as_half(static_cast<unsigned short>(h[e / 2] >> (16 * (e & 1))))), s);
                p.prob[(patch * kPatch + gy) * kPatch + gx] = 1.0f / (1.0f + expf(-s));
            }
        }
        __syncthreads();                                   // TMEM and the planes are free for the next strip
        if (*(volatile int*)&c.fail) break;                // (the same for all: set before the barrier, never cleared)
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kEpiWarps) {
        if (*(volatile int*)&c.fail) {                     // MMAs still in flight end before TMEM goes back
            if (elect_one()) umma_commit(&c.wbar);
            __syncwarp();
            mbar_wait_warp(&c.wbar, 1, p.err, ERR_WAIT_MMA);
        }
        tc_fence_after();
        tmem_dealloc(tm, 256);
    }
}

}  // namespace

cudaError_t launch_rfi_forward_tc(const RfiFwd& p, int n_sm, cudaStream_t s) {
    auto kern = p.A1 ? rfi_forward_kernel<true> : rfi_forward_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem::total);
    if (e != cudaSuccess) return e;
    const int items = p.B * kStrips;
    kern<<<items < 2 * n_sm ? items : 2 * n_sm, kThreadsTc, Smem::total, s>>>(p);
    return cudaGetLastError();
}

}  // namespace gbx
