// The reorder pass of Section 3.2: rays are moved into sorted order.
// out[i] = in[perm[i]].  Reads of `in` are random (one 16-byte lane per field,
// i.e. half a sector); reads of perm and all writes are coalesced.
#include "rr_common.cuh"

namespace rr {

constexpr int kPermuteBlock = 256;
constexpr int kPermuteItems = 2;  // rays per thread: more loads in flight per thread

template <bool PAYLOAD>
__global__ void __launch_bounds__(kPermuteBlock) permute_kernel(const float4 *o_in, const float4 *d_in,
                                                               const uint32_t *p_in, const uint32_t *perm,
                                                               uint32_t n, float4 *o_out, float4 *d_out,
                                                               uint32_t *p_out, uint32_t *err) {
    allow_dependent_launch();
    wait_for_prerequisite();
    const uint32_t base = blockIdx.x * (kPermuteBlock * kPermuteItems) + threadIdx.x;
    uint32_t src[kPermuteItems];
#pragma unroll
    for (int j = 0; j < kPermuteItems; ++j) {
        const uint32_t i = base + j * kPermuteBlock;
        src[j] = i < n ? __ldcs(perm + i) : 0u;
    }
    float4 o[kPermuteItems], d[kPermuteItems];
    uint32_t p[kPermuteItems];
#pragma unroll
    for (int j = 0; j < kPermuteItems; ++j) {
        const uint32_t i = base + j * kPermuteBlock;
        if (i < n && index_ok(src[j], n, err)) {
            o[j] = o_in[src[j]];
            d[j] = d_in[src[j]];
            if (PAYLOAD) p[j] = p_in[src[j]];
        }
    }
#pragma unroll
    for (int j = 0; j < kPermuteItems; ++j) {
        const uint32_t i = base + j * kPermuteBlock;
        if (i < n && (!kChecked || src[j] < n)) {
            o_out[i] = o[j];
            d_out[i] = d[j];
            if (PAYLOAD) p_out[i] = p[j];
        }
    }
}

// Wavefronts too large for L2 are moved one array after the other.  With all
// three at once the random reads touch 36 bytes a ray of source: a sector's
// second ray comes when its sector has left L2, and every 16-byte read costs a
// DRAM access of its own.  One array at a time keeps most of its sectors (133
// MB of origins at 8.3M rays against 129 MB of L2) until their other rays are
// read, for two more streaming reads of the permutation; outputs are written
// evict-first so that they do not push the sources out.  Measured, random
// order with payload: 8.3M rays 0.384 -> 0.254 ms (1.65 -> 2.48 TB/s of the 76
// bytes a ray it cannot do without), 4.1M 0.142 -> 0.090, 3.0M 0.085 -> 0.064;
// pixel-ordered rays, 8.3M: 0.156 -> 0.146.
constexpr int kPhaseItems = 4;  // rays per thread and array

template <typename T>
__device__ __forceinline__ void gather_phase(const T *in, const uint32_t *perm, uint32_t n, T *out,
                                             uint32_t block, uint32_t *err) {
    const uint32_t base = block * (kPermuteBlock * kPhaseItems) + threadIdx.x;
    uint32_t src[kPhaseItems];
    T v[kPhaseItems];
#pragma unroll
    for (int j = 0; j < kPhaseItems; ++j) {
        const uint32_t i = base + j * kPermuteBlock;
        src[j] = i < n ? __ldcs(perm + i) : 0u;
    }
#pragma unroll
    for (int j = 0; j < kPhaseItems; ++j) {
        const uint32_t i = base + j * kPermuteBlock;
        if (i < n && index_ok(src[j], n, err)) v[j] = in[src[j]];
    }
#pragma unroll
    for (int j = 0; j < kPhaseItems; ++j) {
        const uint32_t i = base + j * kPermuteBlock;
        if (i < n && (!kChecked || src[j] < n)) __stcs(out + i, v[j]);
    }
}

__global__ void __launch_bounds__(kPermuteBlock) permute_phased_kernel(
    const float4 *o_in, const float4 *d_in, const uint32_t *p_in, const uint32_t *perm, uint32_t n, float4 *o_out,
    float4 *d_out, uint32_t *p_out, uint32_t phase_blocks, uint32_t *err) {
    wait_for_prerequisite();
    const uint32_t phase = blockIdx.x / phase_blocks, block = blockIdx.x - phase * phase_blocks;
    if (phase == 0)
        gather_phase(o_in, perm, n, o_out, block, err);
    else if (phase == 1)
        gather_phase(d_in, perm, n, d_out, block, err);
    else
        gather_phase(p_in, perm, n, p_out, block, err);
}

// From this many rays on (75 MB of sources, and as much of results) the phases
// pay: at 2.07M rays 0.0455 against 0.0475 ms in random order, at 1.2M 0.0285
// against 0.0265 in pixel order.
constexpr uint32_t kPhasedRays = 1u << 21;

}  // namespace rr

using namespace rr;

extern "C" rr_status rr_permute(const float *o_tmin_in, const float *d_tmax_in, const uint32_t *payload_in,
                                const uint32_t *perm, uint32_t n, float *o_tmin_out, float *d_tmax_out,
                                uint32_t *payload_out, void *stream) {
    if (n == 0) return RR_OK;
    if (!o_tmin_in || !d_tmax_in || !perm || !o_tmin_out || !d_tmax_out)
        return fail(RR_ERR_INVALID_ARG, "rr_permute: NULL buffer");
    if ((payload_in == nullptr) != (payload_out == nullptr))
        return fail(RR_ERR_INVALID_ARG, "rr_permute: payload_in and payload_out must both be set or both NULL");
    if (!aligned16(o_tmin_in) || !aligned16(d_tmax_in) || !aligned16(o_tmin_out) || !aligned16(d_tmax_out) ||
        !aligned(perm, 4) || (payload_in && (!aligned(payload_in, 4) || !aligned(payload_out, 4))))
        return fail(RR_ERR_INVALID_ARG, "rr_permute: misaligned buffer");
    const size_t rb = 16ull * n, pb = 4ull * n;
    if (overlaps(o_tmin_out, rb, o_tmin_in, rb) || overlaps(o_tmin_out, rb, d_tmax_in, rb) ||
        overlaps(d_tmax_out, rb, o_tmin_in, rb) || overlaps(d_tmax_out, rb, d_tmax_in, rb) ||
        overlaps(o_tmin_out, rb, d_tmax_out, rb) || overlaps(o_tmin_out, rb, perm, pb) ||
        overlaps(d_tmax_out, rb, perm, pb) ||
        (payload_in && (overlaps(payload_out, pb, payload_in, pb) || overlaps(payload_out, pb, perm, pb))))
        return fail(RR_ERR_INVALID_ARG, "rr_permute: buffers overlap");
    rr_status st;
    DeviceState *ds = device_state(&st);
    if (!ds) return st;
    cudaStream_t s = as_stream(stream);
    const float4 *oi = reinterpret_cast<const float4 *>(o_tmin_in);
    const float4 *di = reinterpret_cast<const float4 *>(d_tmax_in);
    float4 *oo = reinterpret_cast<float4 *>(o_tmin_out);
    float4 *dd = reinterpret_cast<float4 *>(d_tmax_out);
    uint32_t *err = error_word(ds, s);
    const uint32_t blocks = (n + kPermuteBlock * kPermuteItems - 1) / (kPermuteBlock * kPermuteItems);
    if (n >= kPhasedRays) {
        const uint32_t phase_blocks = (n + kPermuteBlock * kPhaseItems - 1) / (kPermuteBlock * kPhaseItems);
        launch_dependent(permute_phased_kernel, phase_blocks * (payload_in ? 3u : 2u), kPermuteBlock, 0, s, oi, di,
                         payload_in, perm, n, oo, dd, payload_out, phase_blocks, err);
    } else {
        launch_dependent(payload_in ? permute_kernel<true> : permute_kernel<false>, blocks, kPermuteBlock, 0, s, oi, di,
                         payload_in, perm, n, oo, dd, payload_out, err);
    }
    note_launches(1);
    return check_launch("rr_permute");
}
