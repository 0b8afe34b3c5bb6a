// fengine_split.cu -- F-engine launches whose last frame blocks are shared by several CTAs, each with its
// own antennas (fe_plan), and the kernel that adds their beam sums.
#include <algorithm>

#include "fengine_wfft.cuh"

namespace gbx {
namespace {

// The beams of the shared frame blocks, parts added in order: sum of the incoherent sums, and per
// polarisation the detected sum of the voltage sums.  Four channels a thread, stored together where
// `wide`: the beams can be a caller's (corr_integrate_static), at any address of a float.
__global__ void beam_combine_kernel(const FeSplit sp, int n_pol, int n_chan, int first, int n_int, bool wide,
                                    float* __restrict__ beams) {
    const int64_t n = static_cast<int64_t>(sp.frames) * n_chan;
    for (int64_t q = 4 * (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x); q < n;
         q += 4 * static_cast<int64_t>(gridDim.x) * blockDim.x) {
        float4 inc = *reinterpret_cast<const float4*>(sp.inc + q);
        for (int s = 1; s < sp.parts; ++s) {
            const float4 v = *reinterpret_cast<const float4*>(sp.inc + s * n + q);
            inc.x += v.x, inc.y += v.y, inc.z += v.z, inc.w += v.w;
        }
        float pw[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int pol = 0; pol < n_pol; ++pol) {
            float2 c[4] = {};
            for (int s = 0; s < sp.parts; ++s) {
                const float4* v = reinterpret_cast<const float4*>(sp.coh + (static_cast<int64_t>(s) * n_pol + pol) * n + q);
                const float4 u = v[0], w = v[1];
                c[0].x += u.x, c[0].y += u.y, c[1].x += u.z, c[1].y += u.w;
                c[2].x += w.x, c[2].y += w.y, c[3].x += w.z, c[3].y += w.w;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) pw[e] += fmaf(c[e].y, c[e].y, c[e].x * c[e].x);
        }
        float* b = beams + static_cast<int64_t>(first) * n_chan + q;
        float* bc = b + static_cast<int64_t>(n_int) * n_chan;
        if (wide) {
            *reinterpret_cast<float4*>(b) = inc;
            *reinterpret_cast<float4*>(bc) = make_float4(pw[0], pw[1], pw[2], pw[3]);
        } else {
            b[0] = inc.x, b[1] = inc.y, b[2] = inc.z, b[3] = inc.w;
#pragma unroll
            for (int e = 0; e < 4; ++e) bc[e] = pw[e];
        }
    }
}

}  // namespace

FeSplit fe_plan(int n_ant, int n_pol, int n_chan, int n_int, int n_sm) {
    FeSplit sp{};
    if (n_chan > 1024) return sp;
    const int F = 8192 / n_chan, blocks = (n_int + F - 1) / F;
    const int full = blocks / n_sm * n_sm, T = blocks - full;
    // in inputs of a whole CTA's time (3.5 us each): the walk, 3 to fill and drain its pipeline, and for
    // a shared block the partial sums written and read again (40 bytes a point and part at about
    // 5 TB/s) and the launch that adds them
    double best = T ? n_ant * n_pol + 3 : 0;
    const double gain = 0.06 * (blocks / n_sm * (n_ant * n_pol + 3.0) + best);
    best -= gain;
    for (int S = 2; T && S <= std::min(n_ant, 16); ++S) {
        const int rounds = (T * S + n_sm - 1) / n_sm;
        const double cost = rounds * ((n_ant + S - 1) / S * n_pol + 3.0) + 1.0 + T * S * 8192.0 * 40 / 5e12 / 3.5e-6;
        if (cost < best) {
            best = cost;
            sp.full = full;
            sp.parts = S;
            sp.frames = n_int - full * F;
        }
    }
    return sp;
}

size_t fe_split_floats(const FeSplit& sp, int n_pol, int n_chan) {
    return sp.parts > 1 ? static_cast<size_t>(sp.parts) * sp.frames * n_chan * (1 + 2 * n_pol) : 0;
}

FeSplit fe_split_in(FeSplit sp, float* buf, int n_chan) {
    sp.inc = buf;
    sp.coh = reinterpret_cast<float2*>(buf + static_cast<size_t>(sp.parts) * sp.frames * n_chan);
    return sp;
}

cudaError_t launch_fengine_split(const FeParams& p, int mode, const FeSplit& sp, cudaStream_t s) {
    if (p.n_chan * 2 != p.n_fft || sp.parts < 2 || !sp.inc) return cudaErrorInvalidValue;
    cudaError_t e = cudaErrorInvalidValue;
    switch (mode) {
        case OUT_FP32: e = launch_w_mode<OUT_FP32, true>(p, s, &sp); break;
        case OUT_F16: e = launch_w_mode<OUT_F16, true>(p, s, &sp); break;
        case OUT_F32Q: e = launch_w_mode<OUT_F32Q, true>(p, s, &sp); break;
        case OUT_I8B: e = launch_w_mode<OUT_I8B, true>(p, s, &sp); break;
        default: break;
    }
    if (e != cudaSuccess) return e;
    const int64_t quads = static_cast<int64_t>(sp.frames) * p.n_chan / 4;
    // every row of n_chan floats lies as the first one does
    const bool wide = (reinterpret_cast<uintptr_t>(p.beams) & 15) == 0;
    beam_combine_kernel<<<static_cast<int>(std::min<int64_t>((quads + 255) / 256, 4096)), 256, 0, s>>>(
        sp, p.n_pol, p.n_chan, p.n_int - sp.frames, p.n_int, wide, p.beams);
    return cudaGetLastError();
}

}  // namespace gbx
