// The trace's reciprocal and CUDA's rounded one, side by side.
#include <cstdint>

#include "../../paper_2506_11273_gb300/csrc/rr_reciprocal.cuh"

__global__ void both(const float *x, uint32_t n, float *own, float *rounded) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    own[i] = rr::safe_inv(x[i]);
    rounded[i] = __frcp_rn(rr::nonzero_component(x[i]));
}

extern "C" int reciprocals(const float *x, uint32_t n, float *own, float *rounded, void *stream) {
    both<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(x, n, own, rounded);
    return (int)cudaGetLastError();
}
