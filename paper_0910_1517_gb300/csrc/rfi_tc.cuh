// rfi_tc.cuh -- launch interface of the learned flagger's tensor-core forward pass (rfi_tc.cu).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <cstdint>

namespace gbx {

// Packed fp16 weights the forward pass copies into shared memory: the tcgen05 B operands of layers 2
// and 3 (K-major, no swizzle: core matrices of 8 output channels x 8 inputs), tap by tap.
constexpr int kRfiW2Bytes = 9 * 16 * 32 * 2, kRfiW3Bytes = 9 * 32 * 16 * 2;
constexpr int kRfiPackBytes = kRfiW2Bytes + kRfiW3Bytes;
__host__ __device__ constexpr int rfi_pack2(int o, int c, int tap) {
    return tap * 1024 + (c / 8) * 512 + (o / 8) * 128 + (o % 8) * 16 + (c % 8) * 2;
}
__host__ __device__ constexpr int rfi_pack3(int o, int c, int tap) {
    return kRfiW2Bytes + tap * 1024 + (c / 8) * 256 + (o / 8) * 128 + (o % 8) * 16 + (c % 8) * 2;
}

struct RfiFwd {
    const __half* x;           // [B][64][64] patches
    const unsigned char* pack; // kRfiPackBytes of packed weights
    const __half *w1, *b1, *b2, *b3, *w4, *b4;   // w1 [16][9]
    float* prob;               // [B][64][64] probabilities, or nullptr
    __half *A1, *A2, *A3;      // [B][16 | 32 | 16][64][64] activations to keep, or nullptr
    int B;
    unsigned* err;             // device error word
};
cudaError_t launch_rfi_forward_tc(const RfiFwd& p, int n_sm, cudaStream_t s);

}  // namespace gbx
