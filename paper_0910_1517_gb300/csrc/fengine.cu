// fengine.cu -- F-engine of the FX correlator for sm_103a: launches of the kernels in
// fengine_wfft.cuh and fengine_impl.cuh for single integrations, the per-integration phasor
// set-up, the RFI stage's power dumps and the beam averaging.
#include <cmath>
#include <vector>

#include "fengine_wfft.cuh"

namespace gbx {
namespace {
__global__ void phasor_setup_kernel(int n_ant, int n_chan, int n_fft, int n_int, int64_t g0_val,
                                    const int64_t* __restrict__ g0_ptr,
                                    const double* __restrict__ tau, const double* __restrict__ phi0,
                                    const double* __restrict__ rate, float2* __restrict__ pf,
                                    float2* __restrict__ ff, int* __restrict__ D) {
    const int64_t g0 = g0_ptr ? *g0_ptr : g0_val;
    const int64_t id = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    if (id < n_ant) D[id] = model_int_delay(tau[id]);
    if (id / 32 < model_table_warps(n_ant, n_chan, n_int))
        model_table(id / 32, n_ant, n_chan, n_fft, n_int, g0, tau, phi0, rate, pf, ff);
}

__global__ void twiddle_kernel(int n_fft, int count, float2* __restrict__ tw) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < count; e += gridDim.x * blockDim.x) {
        double num, den, sn, cs;
        fengine_tw_angle(n_fft, e, num, den);
        sincospi(2.0 * num / den, &sn, &cs);
        tw[e] = make_float2(static_cast<float>(cs), static_cast<float>(-sn));
    }
}

// Four channels a thread; n sums a dump.  What bounds it: reading the sums, a sixteenth of the
// spectra.  GMRT shape, 60 inputs, 4096 spectra: the whole integration 0.42 ms shorter than with a
// kernel that summed the 2 GB of spectra themselves (0.49 ms).
__global__ void power_dump_kernel(const float4* __restrict__ part, int n, int64_t n_out, int n_quad, float4* __restrict__ P) {
    for (int64_t q = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; q < n_out;
         q += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const float4* src = part + q / n_quad * n * n_quad + q % n_quad;   // dump q / n_quad of all inputs' in order
        float4 a = src[0];
#pragma unroll 4
        for (int j = 1; j < n; ++j) {
            const float4 v = src[static_cast<int64_t>(j) * n_quad];
            a.x += v.x, a.y += v.y, a.z += v.z, a.w += v.w;
        }
        P[q] = a;
    }
}

__global__ void beam_average_kernel(const float* __restrict__ raw, float* __restrict__ out, int n_int, int n_chan,
                                    int beam_avg) {
    const int n_out = n_int / beam_avg;
    const int64_t total = 2LL * n_out * n_chan;
    const float inv = 1.0f / beam_avg;
    for (int64_t q = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; q < total;
         q += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int k = static_cast<int>(q % n_chan);
        const int64_t bt = q / n_chan;
        const int b = static_cast<int>(bt / n_out), to = static_cast<int>(bt % n_out);
        const float* src = raw + (static_cast<int64_t>(b) * n_int + static_cast<int64_t>(to) * beam_avg) * n_chan + k;
        float acc = 0.0f;
        for (int j = 0; j < beam_avg; ++j) acc += src[static_cast<int64_t>(j) * n_chan];
        out[q] = acc * inv;
    }
}

}  // namespace

cudaError_t launch_fengine_twiddles(int n_fft, float2* tw, cudaStream_t s) {
    const int count = fengine_tw_count(n_fft);
    twiddle_kernel<<<(count + 255) / 256, 256, 0, s>>>(n_fft, count, tw);
    return cudaGetLastError();
}

cudaError_t launch_fengine(const FeParams& p, int mode, cudaStream_t s) {
    if (p.n_chan * 2 != p.n_fft) return cudaErrorInvalidValue;
    switch (mode) {
        case OUT_FP32: return launch_w_mode<OUT_FP32, false>(p, s, nullptr);
        case OUT_F16: return launch_w_mode<OUT_F16, false>(p, s, nullptr);
        case OUT_F32Q: return launch_w_mode<OUT_F32Q, false>(p, s, nullptr);
        case OUT_I8B: return launch_w_mode<OUT_I8B, false>(p, s, nullptr);
        default: return cudaErrorInvalidValue;
    }
}

bool fengine_clustered(int n_chan, int mode) {
    return n_chan == 2048 && (mode == OUT_F16 || mode == OUT_I8B);
}

cudaError_t launch_phasor_setup(int n_ant, int n_chan, int n_fft, int n_int, int64_t g0, const double* tau,
                                const double* phi0, const double* rate, float2* pf, float2* ff, int* D,
                                cudaStream_t s, const int64_t* g0_dev) {
    // 64 threads a block: two warps an SM from 152 warps on; at least one warp, so n_ant <= 128 delays too
    const int64_t threads = std::max<int64_t>(32 * model_table_warps(n_ant, n_chan, n_int), n_ant);
    phasor_setup_kernel<<<static_cast<unsigned>((threads + 63) / 64), 64, 0, s>>>(n_ant, n_chan, n_fft, n_int, g0, g0_dev, tau, phi0,
                                                                                 rate, pf, ff, D);
    return cudaGetLastError();
}

cudaError_t launch_power_dumps(const float* part, int n_in, int n_chan, int n_int, int dump, float* P, cudaStream_t s) {
    const int tb = tb_fp32(n_chan), n = dump / tb, n_quad = n_chan / 4;
    if (dump < tb || dump % tb || n_int % dump) return cudaErrorInvalidValue;
    if (n == 1) return cudaSuccess;
    const int64_t n_out = static_cast<int64_t>(n_in) * (n_int / dump) * n_quad;
    const int grid = static_cast<int>(std::min<int64_t>((n_out + 255) / 256, 8192));
    power_dump_kernel<<<grid, 256, 0, s>>>(reinterpret_cast<const float4*>(part), n, n_out, n_quad, reinterpret_cast<float4*>(P));
    return cudaGetLastError();
}

cudaError_t launch_beam_average(const float* raw, float* out, int n_int, int n_chan, int beam_avg,
                                cudaStream_t s) {
    const int64_t total = 2LL * (n_int / beam_avg) * n_chan;
    const int grid = static_cast<int>(std::min<int64_t>((total + 255) / 256, 8192));
    beam_average_kernel<<<grid, 256, 0, s>>>(raw, out, n_int, n_chan, beam_avg);
    return cudaGetLastError();
}

}  // namespace gbx
