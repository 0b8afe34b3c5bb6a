// blank.cu -- statistics of the time-domain voltage blanker (Sec. 5, Eq. 3-4) on sm_103a.
//
// For every (input, block) of raw int8 samples: the median, the MAD (median of |x - med|)
// and the flag threshold of Eq. 4, |x - med| > M MAD / 0.6745.  int8 data make both medians
// exact: the cumulated 256-bin histogram C of x gives the two middle values (their sum is
// 2 med), and the number of deviations d2 = |2x - 2med| up to D is C at the upper end of
// [(2med - D)/2, (2med + D)/2] minus C below its lower end, which gives the two middle
// deviations (their sum is 4 MAD).  The threshold becomes the integer T2 =
// floor(2 M MAD / 0.6745) (computed in FP64), so that a sample is replaced iff d2 > T2 -- the
// same decision as the FP64 comparison -- by rint(sigma g) clamped to +-127, sigma =
// MAD / 0.6745 rounded to FP32 and g the input's table noise at the sample's position.  The
// same CTA then writes the block's blanked samples (testing four samples at a time against
// integer bounds), which the F-engine reads instead of the raw rows.  (Fusing the replacement
// into the F-engine's sample conversion was measured first: +1.75 ms on the GMRT-scale
// F-engine, more than this separate pass.)
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"
#include "fengine.cuh"

namespace gbx {
namespace {

constexpr int kBlankThreads = 256;
constexpr int kBlankWarps = kBlankThreads / 32;
constexpr int kBlankMaxBlock = 32768;     // the list of words to replace holds 16-bit indexes in the histogram's place

// The majority of three bits, bit by bit.
__device__ __forceinline__ uint32_t majority(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a | b)); }

// x + 128 > h for the four int8 of w at once (0 <= h <= 255; h = -1: always), in bit 7 of each byte:
// the seven low bits with `add` carry into bit 7 where they are above h's; an x >= 0 is above any
// h < 128 (`pass` ~0) and an x < 0 above none of the others (`pass` 0).
struct Above {
    uint32_t add, pass;
    __device__ explicit Above(int h)
        : add(static_cast<uint32_t>(h < 128 ? 127 - h : 255 - h) * 0x01010101u), pass(h < 128 ? ~0u : 0u) {}
    __device__ uint32_t operator()(uint32_t w) const { return majority((w & 0x7f7f7f7fu) + add, ~w, pass); }
};

__global__ void __launch_bounds__(kBlankThreads, 6) blank_kernel(const int8_t* __restrict__ x, int64_t ld, int64_t n,
                                                                  int block, double M, const float* __restrict__ noise,
                                                                  int noise_mask, int32_t* __restrict__ stats,
                                                                  int8_t* __restrict__ y, int64_t ldy) {
    // Histogram of the bytes of x, a column of 32-bit counters for each lane: the lanes meet in no
    // bank and a sample costs a shift, a mask and the atomic.  The pass is bound by its accesses to
    // shared memory and its instructions (about 17 a warp's 32 samples).  64 inputs x 8.4e6 samples
    // in blocks of 16384: 290 us, 1.07 GB in and out (363 us with one 256-bin histogram a warp,
    // emulated byte compares and the replacement in place; 16-bit counters or a byte histogram for
    // each thread without atomics were slower: 380 and 690 us).
    __shared__ __align__(16) uint32_t hist[256][32];
    __shared__ int cum[257];               // cum[u]: samples below bin u
    __shared__ int wsum[kBlankWarps];
    __shared__ int mid[4];                 // middle values (bins) and middle deviations, lower and upper
    __shared__ int t2_s, n_words;
    __shared__ float sig_s;
    const int i = blockIdx.y, warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int64_t b = blockIdx.x, p0 = b * block;
    const int len = static_cast<int>(p0 + block <= n ? block : n - p0);
    const int8_t* row = x + static_cast<int64_t>(i) * ld + p0;
    // pass 1: histogram of x (16-byte loads: rows and blocks start on 16-byte boundaries; the next
    // piece is on its way while one is counted).
    const int n16 = len / 16;
    const int4* row16 = reinterpret_cast<const int4*>(row);
    int4 cur = static_cast<int>(threadIdx.x) < n16 ? __ldg(row16 + threadIdx.x) : make_int4(0, 0, 0, 0);
    if (threadIdx.x == 0) n_words = 0;
    for (int q = threadIdx.x; q < 256 * 32 / 4; q += kBlankThreads)
        reinterpret_cast<uint4*>(&hist[0][0])[q] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    const uint32_t col = 4u * lane;
    auto add1 = [&](uint32_t off) {
        atomicAdd(reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned char*>(hist) + ((off & 0x7f80u) | col)), 1u);
    };
    auto count = [&](uint32_t w) {
        add1(w << 7);
        add1(w >> 1);
        add1(w >> 9);
        add1(w >> 17);
    };
    for (int q = threadIdx.x; q < n16; q += kBlankThreads) {
        const int4 next = q + kBlankThreads < n16 ? __ldg(row16 + q + kBlankThreads) : make_int4(0, 0, 0, 0);
        count(static_cast<uint32_t>(cur.x));
        count(static_cast<uint32_t>(cur.y));
        count(static_cast<uint32_t>(cur.z));
        count(static_cast<uint32_t>(cur.w));
        cur = next;
    }
    for (int q = 16 * n16 + threadIdx.x; q < len; q += kBlankThreads) atomicAdd(&hist[static_cast<uint8_t>(row[q])][lane], 1u);
    __syncthreads();
    // thread u adds up the 32 counters of x = u - 128 (16 bytes at a time, the columns rotated by row so that
    // a quarter warp's rows lie in different banks) and the CTA's scan cumulates the bins
    uint32_t c = 0u;
    {
        const uint4* r4 = reinterpret_cast<const uint4*>(&hist[threadIdx.x ^ 128][0]);
#pragma unroll 4
        for (int q = 0; q < 8; ++q) {
            const uint4 v = r4[q ^ (threadIdx.x & 7)];
            c += (v.x + v.y) + (v.z + v.w);
        }
    }
    int incl = static_cast<int>(c);
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kBlankWarps; ++w) incl += w < warp ? wsum[w] : 0;
    if (threadIdx.x == 0) cum[0] = 0;
    cum[threadIdx.x + 1] = incl;
    const int lo = (len - 1) / 2, hi = len / 2;       // the two middle ranks (equal for odd len)
    {
        const int before = incl - static_cast<int>(c);
        if (lo >= before && lo < incl) mid[0] = static_cast<int>(threadIdx.x);
        if (hi >= before && hi < incl) mid[1] = static_cast<int>(threadIdx.x);
    }
    __syncthreads();
    const int med2 = mid[0] + mid[1] - 256;
    // samples x with lo_x <= x <= hi_x
    auto inside = [&](int lo_x, int hi_x) { return cum[min(hi_x, 127) + 129] - cum[max(lo_x, -128) + 128]; };
    {   // pass 2: every d2 has 2 med's parity; thread j holds the j-th such value
        const int D = 2 * static_cast<int>(threadIdx.x) + (med2 & 1);
        const int upto = inside((med2 - D) >> 1, (med2 + D) >> 1);
        const int below = threadIdx.x == 0 ? 0 : inside(((med2 - D) >> 1) + 1, ((med2 + D) >> 1) - 1);
        if (lo >= below && lo < upto) mid[2] = D;
        if (hi >= below && hi < upto) mid[3] = D;
    }
    __syncthreads();
    if (warp == 0) {
        const int mad4 = mid[2] + mid[3];
        const double mad = mad4 / 4.0;
        double t2 = floor(2.0 * (M * mad / 0.6745));
        if (t2 > 1024.0) t2 = 1024.0;
        const int T2 = static_cast<int>(t2);
        if (lane == 0) {
            const int64_t q = static_cast<int64_t>(i) * gridDim.x + b;
            int32_t* st = stats + 4 * q;
            st[0] = med2;
            st[1] = mad4;
            st[2] = T2;
            st[3] = len - inside((med2 - T2 + 1) >> 1, (med2 + T2) >> 1);
            t2_s = T2;
            sig_s = static_cast<float>(mad / 0.6745);
        }
    }
    __syncthreads();
    // pass 3: the blanked block.  |2x - med2| > T2 holds exactly for x > hi_x or x < lo_x,
    // hi_x = floor((med2 + T2) / 2), lo_x = ceil((med2 - T2) / 2) (integer x); clamped to the int8
    // range they compare four samples at a time.  Every piece is copied as it is; the words that
    // hold a flagged sample go on a list and are replaced from it afterwards, a thread a word.
    // (Nearly every warp's 512 samples hold one: replacing it there made the whole warp do all of
    // them.)
    const int T2 = t2_s;
    const float sg = sig_s;
    const int hi_x = min(127, (med2 + T2) >> 1), lo_x = max(-128, (med2 - T2 + 1) >> 1);
    const Above above(hi_x + 128), not_below(lo_x + 127);
    auto flags = [&](uint32_t w) {   // bit 7 of every flagged byte
        return (above(w) | ~not_below(w)) & 0x80808080u;
    };
    const float* g = noise + static_cast<int64_t>(i) * (noise_mask + 1);
    int8_t* out = y + static_cast<int64_t>(i) * ldy + p0;
    auto value = [&](float z) {
        return static_cast<int>(fminf(127.0f, fmaxf(-127.0f, rintf(__fmul_rn(sg, z)))));
    };
    uint16_t* list = reinterpret_cast<uint16_t*>(&hist[0][0]);   // the counters are not needed any more
#pragma unroll 2
    for (int q = threadIdx.x; q < n16; q += kBlankThreads) {
        const int4 v = __ldg(row16 + q);
        reinterpret_cast<int4*>(out)[q] = v;
        const bool f0 = flags(static_cast<uint32_t>(v.x)) != 0u, f1 = flags(static_cast<uint32_t>(v.y)) != 0u;
        const bool f2 = flags(static_cast<uint32_t>(v.z)) != 0u, f3 = flags(static_cast<uint32_t>(v.w)) != 0u;
        if (f0 || f1 || f2 || f3) {
            int at = atomicAdd(&n_words, f0 + f1 + f2 + f3);
            if (f0) list[at++] = static_cast<uint16_t>(4 * q);
            if (f1) list[at++] = static_cast<uint16_t>(4 * q + 1);
            if (f2) list[at++] = static_cast<uint16_t>(4 * q + 2);
            if (f3) list[at++] = static_cast<uint16_t>(4 * q + 3);
        }
    }
    __syncthreads();   // the list is complete, and its words' copies come before their replacement
    for (int t = threadIdx.x; t < n_words; t += kBlankThreads) {
        const int q = list[t];
        const int64_t pos = p0 + 4 * q;
        const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(row) + q), f = flags(w);
        const int64_t at = pos & noise_mask;   // a table of four or more values holds the word's in one piece
        const float4 z = noise_mask >= 3 ? __ldg(reinterpret_cast<const float4*>(g + at))
                                         : make_float4(__ldg(g + at), __ldg(g + ((at + 1) & noise_mask)),
                                                       __ldg(g + ((at + 2) & noise_mask)), __ldg(g + ((at + 3) & noise_mask)));
        const uint32_t lo16 = __byte_perm(value(z.x), value(z.y), 0x0040), hi16 = __byte_perm(value(z.z), value(z.w), 0x0040);
        const uint32_t m = (f >> 7) * 0xffu;
        reinterpret_cast<uint32_t*>(out)[q] = (w & ~m) | (__byte_perm(lo16, hi16, 0x5410) & m);
    }
    auto repl = [&](int64_t pos) { return value(__ldg(g + (pos & noise_mask))); };
    for (int q = 16 * n16 + threadIdx.x; q < len; q += kBlankThreads) {
        const int v = row[q];
        out[q] = static_cast<int8_t>(v > hi_x || v < lo_x ? repl(p0 + q) : v);
    }
}

}  // namespace

cudaError_t launch_blank(const int8_t* x, int64_t ld, int n_in, int64_t n, int block, double M,
                         const float* noise, int noise_mask, int32_t* stats, int8_t* y, int64_t ldy,
                         cudaStream_t s) {
    if (n < 1 || block < 16 || block > kBlankMaxBlock || (block & 15) || (ld & 15) || (ldy & 15)) return cudaErrorInvalidValue;
    const int64_t nb = (n + block - 1) / block;
    if (nb > 2147483647LL || n_in > 65535) return cudaErrorInvalidValue;
    blank_kernel<<<dim3(static_cast<unsigned>(nb), n_in), kBlankThreads, 0, s>>>(x, ld, n, block, M, noise,
                                                                                   noise_mask, stats, y, ldy);
    return cudaGetLastError();
}

}  // namespace gbx
