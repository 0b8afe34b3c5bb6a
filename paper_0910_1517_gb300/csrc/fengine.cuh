// fengine.cuh -- launch interface of the F-engine (integer delay, real FFT,
// Eq. 2 phasor, beams, requantisation) and of the per-integration phasor set-up.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>
#include <cmath>
#include <vector>

namespace gbx {

enum OutMode : int { OUT_FP32 = 0, OUT_F16 = 2, OUT_F32Q = 3, OUT_I8B = 4 };

// Spectra hand-off layout ("K-block layout"), shared by every X-engine:
//   S[k][kb][r][TB]   k channel, kb = t / TB, r = 2*i + c (c = 0 re, 1 im), TB = t % TB
// One (k, kb) block holds every input's rows for TB consecutive frames.
// fp16 (tensor-core X-engine): TB = 8, R = 2 n_in unswizzled rows of 16 bytes -- exactly
// the no-swizzle K-major canonical layout of a tcgen05 operand tile (OUT_F16).  OUT_I8B writes
// the int8 requantised values as bytes in the channel-quad arrangement (i8q_piece) that the
// X-engine gathers by TMA into [kb][r][8 bytes] and widens to fp16 on chip.
// FP32 (CUDA-core X-engine): TB = tb_fp32(n_chan) = 8 frames (4 when an F-engine CTA covers
// only 4 frames, n_chan = 2048), rows padded to Rp = round_up(2 n_in, 8).  The block is cut
// into 16-byte granules of 4 frames of one row, 8 rows (one input group of 4) per row group
// G, and granule g = (r % 8) * TB/4 + (frame % TB) / 4 of group G sits at position
// g ^ (G & 7): the CUDA-core X-engine's threads, which read the same granule of different
// row groups at once, then hit distinct banks, while the re and im rows of one input over
// the TB frames stay one contiguous, aligned 8 * TB-byte piece (the F-engine writes each
// piece in one store instruction).  Padding rows only meet padding inputs, whose products
// are never kept.
constexpr int kTbHalf = 8;

__host__ __device__ constexpr int tb_fp32(int n_chan) { return n_chan >= 2048 ? 4 : 8; }
__host__ __device__ constexpr int rows_fp32(int n_in) { return ((2 * n_in + 7) / 8) * 8; }
// float offset of row r, frame e (0 <= e < tb) inside one FP32 K-block
__host__ __device__ constexpr int fp32_off(int r, int e, int tb) {
    const int G = r >> 3, g = (r & 7) * (tb >> 2) + (e >> 2);
    return G * 8 * tb + ((g ^ (G & 7)) << 2) + (e & 3);
}

// FP32 spectra in the channel-quad layout (OUT_F32Q, the F-to-X hand-off of CORR_FP32TC for
// n_chan <= 1024): the piece of channel k, 8-frame K-block kb and input i -- 8 re then 8 im FP32
// values, 64 bytes -- at float offset
//   (((k / 4) * ntb + kb) * n_in + i) * 64 + (k % 4) * 16
// i.e. [k / 4][kb][i][k % 4][16]: the F-engine, which holds one input of 8 frames for every
// channel, writes 256 contiguous bytes per channel quad (instead of 64-byte pieces 4 MB apart,
// which leave its stores at a third of the HBM bandwidth), and a channel's stage is a strided
// gather that one 5-D TMA tensor copy performs ([kb][i][16] = [kb][row 2i + c][8 frames]).
__host__ __device__ constexpr int64_t f32q_piece(int k, int64_t kb, int i, int64_t ntb, int n_in) {
    return (((static_cast<int64_t>(k) >> 2) * ntb + kb) * n_in + i) * 64 + (k & 3) * 16;
}
// The same channel-quad arrangement for the int8 bytes of OUT_I8B: the piece of (k, kb, i) -- 8 re
// then 8 im bytes, 16 bytes -- at byte offset (((k / 4) * ntb + kb) * n_in + i) * 64 + (k % 4) * 16,
// so that four consecutive channels' pieces make whole 64-byte runs.
__host__ __device__ constexpr int64_t i8q_piece(int k, int64_t kb, int i, int64_t ntb, int n_in) {
    return f32q_piece(k, kb, i, ntb, n_in);
}

struct FeParams {
    const int8_t* x;       // input rows, row i at x + i*ld
    int64_t ld;            // row stride in bytes (multiple of 16)
    int64_t n_avail;       // readable samples per row
    int n_ant, n_pol, n_in, n_fft, n_chan, n_int;
    const int* D;          // [n_ant] integer delays
    const float2* pf;      // [n_ant][n_chan] fractional-delay phasor exp(+2 pi i k tau_f / N)
    const float2* ff;      // [n_ant][n_int] fringe phasor exp(-i phi_a(g0 + t))
    const float2* wcoh;    // [n_ant][n_chan] coherent-beam weight g_a exp(i theta_ak), 0 if unselected
    const float* ginc;     // [n_ant] incoherent weight g_a^2, 0 if unselected
    union {                // (a field of its own for the dumps made every kernel here spill)
        const float* scale;   // I8 / F16: [n_in][n_chan] requantisation scales
        float* dump;          // FP32 forms: |Y|^2 summed over each K-block's frames
                              // [n_in][n_int / tb][n_chan], or nullptr
    };
    void* spec;            // spectra in the K-block layout
    float* beams;          // [2][n_int][n_chan] raw-resolution beams (0 inc, 1 coh)
    const float2* tw;      // FFT twiddles laid out as fengine_tw_angle() describes
    unsigned* err;
};

// Sub-arrays of one batch (corr_batch_*).
constexpr int kMaxSub = 8;

// Twiddle table of the F-engines for n_fft (M = n_fft / 2); entry e holds exp(-2 pi i num / den)
// (fengine_tw_angle), evaluated in FP64 on the device and rounded once (launch_fengine_twiddles).
//   part A, read by the kernel of fengine_impl.cuh (n_fft = 4096): [R2][16]
//     pass-2 twiddles W_{16 R2}^(j r), [R3][16 R2] pass-3 twiddles W_M^(j r) when R3 > 1, then
//     [M/2 + 1] real-split twiddles W_N^k;
//   part B (M <= 1024), read by the warp-FFT kernel of fengine_wfft.cuh: [P/2][32][2] inter-pass
//     twiddles W_M^(l k1) (k1 = 2 j + b at [j][l][b]; P = M/32; at P = 1 its 32 entries are
//     unused), then [M/2 + 1] W_N^k.
__host__ __device__ constexpr int fengine_tw_r2(int M) { return (M / 16 >= 16) ? 16 : M / 16; }
__host__ __device__ constexpr int fengine_tw_r3(int M) { return M / (16 * fengine_tw_r2(M)); }
__host__ __device__ constexpr int fengine_tw_a_count(int n_fft) {
    return fengine_tw_r2(n_fft / 2) * 16 +
           (fengine_tw_r3(n_fft / 2) > 1 ? fengine_tw_r3(n_fft / 2) * 16 * fengine_tw_r2(n_fft / 2) : 0) + n_fft / 4 + 1;
}
__host__ __device__ constexpr int fengine_tw_wfft_offset(int n_fft) { return fengine_tw_a_count(n_fft); }
__host__ __device__ constexpr int fengine_tw_count(int n_fft) {
    return fengine_tw_a_count(n_fft) + (n_fft / 2 <= 1024 ? (n_fft / 64) * 32 + n_fft / 4 + 1 : 0);
}
__host__ __device__ inline void fengine_tw_angle(int n_fft, int e, double& num, double& den) {
    const int M = n_fft / 2, R2 = fengine_tw_r2(M), R3 = fengine_tw_r3(M), Ns3 = 16 * R2;
    const int A = fengine_tw_a_count(n_fft);
    if (e < A) {
        if (e < R2 * 16) {                                   // pass 2: W_{16 R2}^(j r), [r][j]
            num = static_cast<double>(e % 16) * (e / 16);
            den = 16.0 * R2;
            return;
        }
        e -= R2 * 16;
        if (R3 > 1 && e < R3 * Ns3) {                        // pass 3: W_M^(j r), [r][j]
            num = static_cast<double>(e % Ns3) * (e / Ns3);
            den = M;
            return;
        }
        e -= (R3 > 1 ? R3 * Ns3 : 0);                        // real split: W_N^k
        num = e;
        den = n_fft;
        return;
    }
    e -= A;
    if (e < (M / 32) * 32) {                                 // inter-pass: W_M^(l k1), [k1 / 2][l][k1 % 2]
        const int l = (e >> 1) & 31, k1 = ((e >> 6) << 1) + (e & 1);
        num = static_cast<double>(l) * k1;
        den = M;
        return;
    }
    num = e - (M / 32) * 32;                                 // real split: W_N^k
    den = n_fft;
}
cudaError_t launch_fengine_twiddles(int n_fft, float2* tw, cudaStream_t s);

// int8 pair (x[2n], x[2n+1]) as the complex sample z[n], without the conversion unit: each byte
// b, offset to b + 128 (sign bit flipped), becomes the low byte of the float 2^23 + b + 128
// (exponent byte 0x4B), and one packed subtraction of 2^23 + 128 leaves b exactly
__device__ __forceinline__ float2 pair_u16(uint32_t w) {
    const uint32_t x = w ^ 0x8080u;
    const uint32_t lo = __byte_perm(x, 0x4B000000u, 0x7440), hi = __byte_perm(x, 0x4B000000u, 0x7441);
    return __fadd2_rn(make_float2(__uint_as_float(lo), __uint_as_float(hi)), make_float2(-8388736.0f, -8388736.0f));
}

// The per-antenna delay model (Sec. 2.1, Eq. 2), shared by every table set-up:
// integer delay D = floor(tau + 1/2), fractional-delay (FSTC) phasor exp(+2 pi i k tau_f / N)
// with tau_f = tau - D, fringe phasor exp(-i phi) with phi = phi0 + rate g over the global frame
// count g, reduced mod 2 pi in FP64.
__host__ __device__ inline int model_int_delay(double tau) { return static_cast<int>(floor(tau + 0.5)); }
struct cplx64 {
    double re, im;
};
__device__ inline cplx64 model_fstc(double tau, int k, int n_fft) {
    const double tf = tau - floor(tau + 0.5);
    cplx64 c;
    sincospi(2.0 * k * tf / n_fft, &c.im, &c.re);
    return c;
}
__device__ inline cplx64 model_fringe(double phi0, double rate, int64_t g) {
    const double twopi = 6.283185307179586476925286766559;
    double ph = phi0 + rate * static_cast<double>(g);
    ph -= twopi * rint(ph / twopi);
    cplx64 c;
    sincos(ph, &c.im, &c.re);
    c.im = -c.im;
    return c;
}
// The phasor tables pf [n_ant][n_chan] (model_fstc) and ff [n_ant][n_int] (model_fringe of frame g0 +
// t), rounded once to FP32.  A warp takes 512 consecutive entries of one antenna: phasor 32 q + l is
// the FP64 product of entry 32 q (lane q's sine and cosine) and of l steps from it (lane l's), so that
// an entry costs four FP64 multiply-adds instead of a sine and cosine of some sixty -- FP64 runs at a
// sixty-fourth of FP32 here.  32 antennas x (1024 channels + 8192 frames): 25 -> 10.5 us.  Up to 98304
// entries in all a warp takes 32 and every lane its own sine and cosine: that many warps fill the SMs
// evenly and take one such latency instead of two (16 x (512 + 4096): 8.8 us and 10.3; 4 x (256 + 64): 4.8, 5.8 in 256-thread
// blocks).
__host__ __device__ inline int model_tile(int n_ant, int n_chan, int n_int) {
    return static_cast<int64_t>(n_ant) * (n_chan + n_int) <= 98304 ? 32 : 512;
}
__host__ __device__ inline int64_t model_table_warps(int n_ant, int n_chan, int n_int) {
    const int t = model_tile(n_ant, n_chan, n_int);
    return static_cast<int64_t>(n_ant) * ((n_chan + t - 1) / t + (n_int + t - 1) / t);
}
__device__ inline void model_table(int64_t warp, int n_ant, int n_chan, int n_fft, int n_int, int64_t g0, const double* tau,
                                   const double* phi0, const double* rate, float2* pf, float2* ff) {
    const int lane = threadIdx.x & 31, t = model_tile(n_ant, n_chan, n_int);
    const int tp = (n_chan + t - 1) / t, per = tp + (n_int + t - 1) / t;
    const int a = static_cast<int>(warp / per), tile = static_cast<int>(warp % per);
    const bool fstc = tile < tp;
    const int e0 = t * (fstc ? tile : tile - tp), n = min(t, (fstc ? n_chan : n_int) - e0);
    const int step = t == 32 ? 1 : 32;
    const cplx64 E = fstc ? model_fstc(tau[a], e0 + step * lane, n_fft) : model_fringe(phi0[a], rate[a], g0 + e0 + step * lane);
    float2* out = (fstc ? pf + static_cast<int64_t>(a) * n_chan : ff + static_cast<int64_t>(a) * n_int) + e0 + lane;
    if (step == 1) {
        if (lane < n) *out = make_float2(static_cast<float>(E.re), static_cast<float>(E.im));
        return;
    }
    const cplx64 R = fstc ? model_fstc(tau[a], lane, n_fft) : model_fringe(0.0, rate[a], lane);
#pragma unroll 4
    for (int q = 0; q < 16; ++q) {
        const double er = __shfl_sync(0xffffffffu, E.re, q), ei = __shfl_sync(0xffffffffu, E.im, q);
        if (32 * q + lane < n)
            out[32 * q] = make_float2(static_cast<float>(er * R.re - ei * R.im), static_cast<float>(er * R.im + ei * R.re));
    }
}

cudaError_t launch_fengine(const FeParams& p, int mode, cudaStream_t s);

// Frame blocks shared by several CTAs (n_chan <= 1024).  A CTA walks every input of its frame block, so
// an integration takes whole rounds of the SMs: 2 blocks of a tiny one leave 150 idle, 512 blocks on
// 152 SMs take four rounds for 3.4.  The blocks of the last, partial round are therefore cut into
// `parts` CTAs that take n_ant / parts antennas each, where that shortens the launch (fe_plan, by
// more than 6 % of the whole); their beam sums go to inc [parts][frames][n_chan] and coh
// [parts][n_pol][frames][n_chan], from where one kernel adds them.  Measured, whole integrations:
// 4 antennas x 64 spectra of 512 points 64 -> 49 us (2 blocks, 4 parts), 60 antennas x 160 of 256
// points 484 -> 103 us (3 blocks), 16 antennas x 1488 of 2048 points 460 -> 325 us (186 blocks, 34
// of them shared), 32 antennas x 4096 behind the blanker 1.76 -> 1.66 ms (512 blocks, 56 shared).
struct FeSplit {
    int full = 0;          // blocks of the full rounds: whole CTAs, the first ones
    int parts = 0;         // CTAs a block after them (0 or 1: nothing is shared)
    int frames = 0;        // frames of the shared blocks
    float* inc = nullptr;
    float2* coh = nullptr;
};
FeSplit fe_plan(int n_ant, int n_pol, int n_chan, int n_int, int n_sm);     // without buffers
size_t fe_split_floats(const FeSplit& sp, int n_pol, int n_chan);           // floats of its buffers
FeSplit fe_split_in(FeSplit sp, float* buf, int n_chan);                     // ... placed at buf (16-byte aligned)
cudaError_t launch_fengine_split(const FeParams& p, int mode, const FeSplit& sp, cudaStream_t s);
// true where launch_fengine launches 2-CTA clusters (n_chan 2048, fp16 layouts and int8 bytes)
bool fengine_clustered(int n_chan, int mode);

// pf, ff and D for one integration from the FP64 delay / fringe model.
// g0_dev, when given, is read on the device instead of g0 (graph-captured launches).
cudaError_t launch_phasor_setup(int n_ant, int n_chan, int n_fft, int n_int, int64_t g0, const double* tau,
                                const double* phi0, const double* rate, float2* pf, float2* ff, int* D,
                                cudaStream_t s, const int64_t* g0_dev = nullptr);

// Auto-power dumps from the F-engine's K-block sums (FeParams::dump, [n_in][n_int / tb][n_chan], tb =
// tb_fp32(n_chan)): P[i][d][k] = sum of |Y_i[t][k]|^2 over the `dump` frames of dump d, dump a
// multiple of tb dividing n_int (with dump = tb the sums are the dumps, and nothing is launched).
cudaError_t launch_power_dumps(const float* part, int n_in, int n_chan, int n_int, int dump, float* P, cudaStream_t s);

// Time-domain voltage blanker (blank.cu, Sec. 5, Eq. 3-4) on rows x[i][0..n) cut into blocks of
// `block` samples (a multiple of 16): per block, stats [n_in][ceil(n / block)][4] = 2 med, 4 MAD,
// T2 = floor(2 M MAD / 0.6745) and the number of samples with |2x - 2 med| > T2, and the blanked
// rows y[i][0..n) (stride ldy): flagged samples replaced by rint(sigma g[i][pos & noise_mask])
// clamped to +-127, sigma = MAD / 0.6745 rounded to FP32; the rest copied.
cudaError_t launch_blank(const int8_t* x, int64_t ld, int n_in, int64_t n, int block, double M,
                         const float* noise, int noise_mask, int32_t* stats, int8_t* y, int64_t ldy,
                         cudaStream_t s);

// Phased beams with full-polar products or voltages (multibeam.cu) from the FP32 spectra:
// w [n_chan][wstride] float2, entry b * n_ant + a the weight of antenna a in beam b for the channel
// (wstride = multibeam_wstride(): n_beams * n_ant rounded up to even); out [n_beams][n_int/avg][n_chan]
// float4.  avg a power of two, max(64, avg) dividing n_int; products 1 (voltages) needs avg = 1.
int multibeam_max_beams();
int multibeam_wstride(int n_beams, int n_ant);
cudaError_t launch_multibeam(const float* spec, int n_ant, int n_pol, int n_chan, int n_int, const float2* w,
                             int n_beams, int products, int avg, float4* out, unsigned* err, cudaStream_t s);

// The same phased beams on the tcgen05 tensor cores (multibeam_tc.cu): FP32 accuracy from an
// on-chip fp16 hi/lo split of weights and spectra; n_ant <= 64, n_beams <= 64, n_int % 64 == 0.
// launch_multibeam takes this form for more than 24 beams where it applies.  split_scale: power of two bringing the
// spectra below the fp16 range (2^-(log2 n_fft - 8)).
bool multibeam_tc_supported(int n_ant, int n_pol, int n_chan, int n_int);
cudaError_t launch_multibeam_tc(const float* spec, int n_ant, int n_pol, int n_chan, int n_int, const float2* w,
                                int wstride, int n_beams, int products, int avg, float split_scale, float4* out,
                                unsigned* err, cudaStream_t s);

// ADC-format 4-bit ingest (ingest4.cu): card rows packed[c][0..2n) (stride ld, even) -> int8 rows
// rows[4c + j][0..n) (stride ldr), the 4 interleaved inputs of each card demultiplexed and sign-extended.
cudaError_t launch_unpack4(const uint8_t* packed, int64_t ld, int n_cards, int64_t n, int8_t* rows, int64_t ldr,
                           int n_sm, cudaStream_t s);

// beams_out[b][to][k] = mean over beam_avg frames of beams_raw[b][to*beam_avg + j][k]
cudaError_t launch_beam_average(const float* raw, float* out, int n_int, int n_chan, int beam_avg,
                                cudaStream_t s);

}  // namespace gbx
