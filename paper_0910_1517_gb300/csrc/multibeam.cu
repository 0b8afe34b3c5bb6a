// multibeam.cu -- several phased-array beams with full-polar products or voltages (Sec. 2.2:
// the coherent beamformer also gives the voltage cross products for the Stokes parameters;
// Sec. 5: multiple phased beams covering different directions in the primary beam), from the
// F-engine's FP32 spectra:
//   U_bp[t][k] = sum_a w[k][b][a] Y_{a,p}[t][k]     (FP32 complex multiply-adds)
//   full polar (products 0): mean over `avg` frames of |U_b0|^2, |U_b1|^2, Re U_b0 conj U_b1,
//                            Im U_b0 conj U_b1
//   voltages   (products 1, avg 1): Re U_b0, Im U_b0, Re U_b1, Im U_b1
//
// A CTA takes channel k and `span` frames, 128 at a time.  A stage's FP32 K-blocks land as they are,
// one bulk copy a K-block at a pitch that spreads consecutive K-blocks over the banks, so that lane
// (K-block, granule) reads its 16 bytes -- four consecutive frames of one row -- without conflicts
// and without transposing the stage.  A thread forms BPT beams of its four frames, two frames a
// packed FP32x2 operation: four 16-byte sample reads and BPT 8-byte weight reads an antenna serve
// 16 BPT packed multiply-adds.  Warps take beam groups.  A window of `avg` frames is summed in the
// lane, by shuffles across its lanes and then across stages in order.  One buffer a CTA; the SM's
// other CTAs compute while one waits for its copy.
// What bounds it: the FP32 pipe from about 8 beams on, the read of the spectra below.  GMRT shape,
// 4096 spectra, 16 beams, 256-frame windows: 0.76 ms (2.15 GB in, 0.49 ms of multiply-adds); 1.67 ms with the stage transposed
// through shared memory and two beams a thread (six shared-memory reads for 16 multiply-adds).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "common.cuh"
#include "fengine.cuh"

namespace gbx {
namespace {

constexpr int kMbMaxBeams = 64;                 // beams per launch
constexpr int kMbFrames = 128;                  // frames per shared-memory stage (four a lane)
constexpr int kMbMaxIn = 128;
constexpr int kMbTcMinBeams = 24;               // more beams than this: the tensor-core form

// bytes from one K-block of tb frames to the next in shared memory: the K-blocks of a
// quarter warp's lanes (16 bytes each; two lanes a K-block at tb 8) fall into different banks
__host__ __device__ constexpr int mb_pitch(int n_in, int tb) { return rows_fp32(n_in) * tb * 4 + 4 * tb; }
__host__ __device__ constexpr int mb_stage_bytes(int n_in, int tb) { return (kMbFrames / tb) * mb_pitch(n_in, tb); }

template <int BPT, int TB>   // beams per thread, frames per K-block
__global__ void __launch_bounds__(512) multibeam_kernel(const float* __restrict__ spec, int n_ant, int n_pol, int n_chan,
                                                        int n_int, const float2* __restrict__ w, int wstride, int n_beams,
                                                        int products, int avg, int span, float4* __restrict__ out, unsigned* err) {
    extern __shared__ __align__(128) unsigned char smb[];
    __shared__ __align__(8) uint64_t bar;
    constexpr int H = TB / 4;                                       // granules of a row in a K-block
    const int n_in = n_ant * n_pol, pitch = mb_pitch(n_in, TB);
    const float2* ws = reinterpret_cast<const float2*>(smb + mb_stage_bytes(n_in, TB));   // [beam][antenna] of channel k
    const int k = blockIdx.x, t0 = blockIdx.y * span;
    const int64_t ntb = n_int / TB;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const uint32_t kb_bytes = static_cast<uint32_t>(rows_fp32(n_in)) * TB * 4;
    const int n_stage = (span + kMbFrames - 1) / kMbFrames;
    auto issue = [&](int st) {   // warp 0: stage st's K-blocks, and with the first the channel's weights
        const int kbs = min(kMbFrames, span - st * kMbFrames) / TB;
        if (lane == 0) {
            mbar_arrive_expect_tx(&bar, kbs * kb_bytes + (st == 0 ? wstride * static_cast<uint32_t>(sizeof(float2)) : 0u));
            if (st == 0)
                bulk_g2s(const_cast<float2*>(ws), w + static_cast<int64_t>(k) * wstride, wstride * sizeof(float2), &bar);
        }
        __syncwarp();
        const float* src = spec + (static_cast<int64_t>(k) * ntb + (t0 + st * kMbFrames) / TB) * (kb_bytes / 4);
        for (int q = lane; q < kbs; q += 32) bulk_g2s(smb + q * pitch, src + static_cast<int64_t>(q) * (kb_bytes / 4), kb_bytes, &bar);
    };
    if (tid == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (warp == 0) issue(0);
    const int n_out = n_int / avg, b0 = warp * BPT;
    const unsigned char* mine = smb + (lane / H) * pitch;           // this lane's K-block, granule lane % H of each row
    float4 acc[BPT];                                                // windows of more than a stage (lane 0)
#pragma unroll
    for (int q = 0; q < BPT; ++q) acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int st = 0; st < n_stage; ++st) {
        if (!__syncthreads_and(mbar_wait_warp(&bar, st & 1, err, ERR_WAIT_STAGE))) {
            if (tid == 0) mbar_wait(&bar, st & 1, nullptr, 0);      // the copies in flight land before the CTA exits (bounded)
            break;
        }
        const int frames = min(kMbFrames, span - st * kMbFrames);
        const bool live = 4 * lane < frames;                        // (a last stage of 64 frames: half the lanes)
        float2 ur[BPT][2][2], ui[BPT][2][2];                        // [beam][pol][frames 0, 1 | 2, 3]
#pragma unroll
        for (int q = 0; q < BPT; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) ur[q][e / 2][e % 2] = ui[q][e / 2][e % 2] = make_float2(0.f, 0.f);
        for (int a = 0; a < n_ant; ++a) {
            float4 yr[2], yi[2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                // rows 2i and 2i + 1 of input i: granules ((r % 8) H + half) ^ (G % 8) of row group G
                const int i = a * n_pol + (p < n_pol ? p : 0), G = i >> 2, g = (2 * i) & 7;
                const unsigned char* grp = mine + G * 128 * H;
                yr[p] = *reinterpret_cast<const float4*>(grp + (((g * H + lane % H) ^ (G & 7)) << 4));
                yi[p] = *reinterpret_cast<const float4*>(grp + ((((g + 1) * H + lane % H) ^ (G & 7)) << 4));
            }
#pragma unroll
            for (int q = 0; q < BPT; ++q) {
                const float2 wv = ws[(b0 + q < n_beams ? b0 + q : 0) * n_ant + a];
                const float2 wr = make_float2(wv.x, wv.x), wi = make_float2(wv.y, wv.y), nwi = make_float2(-wv.y, -wv.y);
#pragma unroll
                for (int p = 0; p < 2; ++p)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float2 r = h ? make_float2(yr[p].z, yr[p].w) : make_float2(yr[p].x, yr[p].y);
                        const float2 m = h ? make_float2(yi[p].z, yi[p].w) : make_float2(yi[p].x, yi[p].y);
                        ur[q][p][h] = __ffma2_rn(wr, r, __ffma2_rn(nwi, m, ur[q][p][h]));
                        ui[q][p][h] = __ffma2_rn(wr, m, __ffma2_rn(wi, r, ui[q][p][h]));
                    }
            }
        }
        __syncthreads();                                            // the stage is read: the next may land
        if (warp == 0 && st + 1 < n_stage) {
            fence_proxy_async_smem();
            issue(st + 1);
        }
        const int ts = t0 + st * kMbFrames + 4 * lane;              // this lane's first frame
#pragma unroll
        for (int q = 0; q < BPT; ++q) {
            const int b = b0 + q;
            if (b >= n_beams) break;                                // (the same for the whole warp)
            float4* ob = out + static_cast<int64_t>(b) * n_out * n_chan + k;
            float4 v[4];
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                auto at = [&](const float2 (&u)[2][2], int p) { return (f & 1) ? u[p][f / 2].y : u[p][f / 2].x; };
                const float r0 = at(ur[q], 0), i0 = at(ui[q], 0), r1 = n_pol == 2 ? at(ur[q], 1) : 0.0f, i1 = n_pol == 2 ? at(ui[q], 1) : 0.0f;
                v[f] = products == 1 ? make_float4(r0, i0, r1, i1)
                                     : make_float4(r0 * r0 + i0 * i0, r1 * r1 + i1 * i1, r0 * r1 + i0 * i1, i0 * r1 - r0 * i1);
            }
            auto add = [](float4 x, float4 y) { return make_float4(x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w); };
            const float sc = 1.0f / avg;
            auto put = [&](int t, float4 x) { ob[static_cast<int64_t>(t / avg) * n_chan] = make_float4(x.x * sc, x.y * sc, x.z * sc, x.w * sc); };
            if (avg <= 2) {
                if (live) {
                    if (avg == 1) {
#pragma unroll
                        for (int f = 0; f < 4; ++f) put(ts + f, v[f]);
                    } else {
                        put(ts, add(v[0], v[1]));
                        put(ts + 2, add(v[2], v[3]));
                    }
                }
                continue;
            }
            float4 s = add(add(v[0], v[1]), add(v[2], v[3]));
            if (!live) s = make_float4(0.f, 0.f, 0.f, 0.f);
            const int lanes = min(avg / 4, 32);
            for (int off = 1; off < lanes; off <<= 1) {
                s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
                s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
                s.z += __shfl_xor_sync(0xffffffffu, s.z, off);
                s.w += __shfl_xor_sync(0xffffffffu, s.w, off);
            }
            if (avg <= kMbFrames) {
                if (live && lane % lanes == 0) put(ts, s);
            } else {                                                // stages of one window, in order
                acc[q] = add(acc[q], s);
                if ((st + 1) * kMbFrames % avg == 0) {
                    if (lane == 0) put(ts, acc[q]);
                    acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
        }
    }
}

}  // namespace

int multibeam_max_beams() { return kMbMaxBeams; }

int multibeam_wstride(int n_beams, int n_ant) { return ((n_beams * n_ant + 1) / 2) * 2; }

cudaError_t launch_multibeam(const float* spec, int n_ant, int n_pol, int n_chan, int n_int, const float2* w,
                             int n_beams, int products, int avg, float4* out, unsigned* err, cudaStream_t s) {
    if (n_beams < 1 || n_beams > kMbMaxBeams || avg < 1 || (avg & (avg - 1)) || n_int % (avg > 64 ? avg : 64) ||
        (products != 0 && products != 1) || (products == 1 && avg != 1) || n_ant * n_pol > kMbMaxIn)
        return cudaErrorInvalidValue;
    // frames per CTA: a multiple of avg dividing n_int, of 128 where there are as many, up to 512
    // (its later stages' copies run while the earlier ones' products are formed)
    int span = avg > 64 ? avg : 64;
    while (span < 512 && n_int % (2 * span) == 0) span *= 2;
    const int wstride = multibeam_wstride(n_beams, n_ant);
    // the tensor-core form for many beams: its time hardly depends on their count (1.7 ms for 64 beams
    // at GMRT scale, 8192 spectra), the CUDA-core kernel's grows with it (1.5 ms for 16, 2.0 ms for
    // 24), but its fp16 hi/lo split is less exact (errors of 5e-7 to 4e-6 against 1e-7 to 3e-6), so
    // the line stays above the crossing
    if (n_beams > kMbTcMinBeams && multibeam_tc_supported(n_ant, n_pol, n_chan, n_int)) {
        int e = -8;
        for (int n = 2 * n_chan; n > 1; n >>= 1) ++e;
        return launch_multibeam_tc(spec, n_ant, n_pol, n_chan, n_int, w, wstride, n_beams, products, avg,
                                   ldexpf(1.0f, -e), out, err, s);
    }
    const int tb = tb_fp32(n_chan), n_in = n_ant * n_pol;
    const size_t smem = static_cast<size_t>(mb_stage_bytes(n_in, tb)) + sizeof(float2) * wstride;
    const dim3 grid(n_chan, n_int / span);
    auto go = [&](auto kern, int bpt) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        if (e != cudaSuccess) return e;
        kern<<<grid, 32 * ((n_beams + bpt - 1) / bpt), smem, s>>>(spec, n_ant, n_pol, n_chan, n_int, w, wstride, n_beams, products,
                                                                 avg, span, out, err);
        return cudaGetLastError();
    };
    // beams a thread: four keep the FP32 pipe ahead of the shared-memory reads; fewer beams than 16
    // take less, so that a CTA has four warps
    if (tb == 8) return n_beams > 8 ? go(multibeam_kernel<4, 8>, 4) : n_beams > 4 ? go(multibeam_kernel<2, 8>, 2) : go(multibeam_kernel<1, 8>, 1);
    return n_beams > 8 ? go(multibeam_kernel<4, 4>, 4) : n_beams > 4 ? go(multibeam_kernel<2, 4>, 2) : go(multibeam_kernel<1, 4>, 1);
}

}  // namespace gbx
