// The reorder pass of Section 3.2: rays are moved into sorted order.
// out[i] = in[perm[i]].  Reads of `in` are random (one 16-byte lane per field,
// i.e. half a sector); reads of perm and all writes are coalesced.
#include "rr_common.cuh"

namespace rr {

constexpr int kPermuteBlock = 256;
constexpr int kPermuteItems = 2;  // rays per thread: more loads in flight per thread
constexpr uint32_t kPermuteRays = kPermuteBlock * kPermuteItems;

// Wavefronts too large for L2 are moved one array after the other.  With all
// three at once the random reads touch 36 bytes a ray of source: a sector's
// second ray comes when its sector has left L2, and every 16-byte read costs a
// DRAM access of its own.  One array at a time keeps most of its sectors (133
// MB of origins at 8.3M rays against 129 MB of L2) until their other rays are
// read, for two more streaming reads of the permutation; outputs are written
// evict-first so that they do not push the sources out.  The payload goes first:
// it leaves room for the permutation, which the next array then finds in L2.
// A tile of the permutation is moved in ROUNDS rounds of PER rays a thread, and
// one array of it takes a block as long as all arrays of kPermuteRays rays.
template <bool PAYLOAD>
struct PhaseTile {
    static constexpr int kPhases = PAYLOAD ? 3 : 2, PER = PAYLOAD ? 3 : 4, ROUNDS = PAYLOAD ? 2 : 1;
    static constexpr uint32_t kRays = kPermuteBlock * PER * ROUNDS;
    static_assert(kRays == kPhases * kPermuteRays, "a tile's phases share its rays when they are moved at once");
};

// Whether a warp's 32 rays are in order already, or nearly: their sources lie
// within 40 rays of one another, so their sectors are used up at once and phases
// would only read the permutation three times.  Sparser runs of sources, as coarse
// keys of ordered rays leave them, are better moved in phases: 16-bit Aila keys of
// 8.3M pixel-ordered rays 111 us with the line at 40, 116 at 64, 127 at 128.
__device__ __forceinline__ bool row_in_order(uint32_t src) {
    return __reduce_max_sync(0xFFFFFFFFu, src) - __reduce_min_sync(0xFFFFFFFFu, src) < 40u;
}

// One array of a tile.  ORDER: true, and nothing is moved, where the warp's first
// row of the tile is in order; every array's block reads that row and finds the
// same.
template <int PER, int ROUNDS, bool KEEP, bool ORDER, typename T>
__device__ __forceinline__ bool gather_phase(const T *in, const uint32_t *perm, uint32_t n, T *out, uint32_t first,
                                             uint32_t *err) {
#pragma unroll 1
    for (int q = 0; q < ROUNDS; ++q) {
        const uint32_t base = first + q * (kPermuteBlock * PER) + threadIdx.x;
        uint32_t src[PER];
        T v[PER];
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const uint32_t i = base + j * kPermuteBlock;
            src[j] = i < n ? (KEEP ? perm[i] : __ldcs(perm + i)) : 0u;
        }
        if (ORDER && q == 0 && (base | 31u) < n && row_in_order(src[0])) return true;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const uint32_t i = base + j * kPermuteBlock;
            if (i < n && index_ok(src[j], n, err)) v[j] = in[src[j]];
        }
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const uint32_t i = base + j * kPermuteBlock;
            if (i < n && (!kChecked || src[j] < n)) __stcs(out + i, v[j]);
        }
    }
    return false;
}

// A block moves kPermuteRays rays, every array of them; PHASED: one array of a
// tile, but for warps whose rays are in order: they move every array of their
// share of the tile (with a payload; without one, two readings of the permutation
// are not worth the question).
// early: the next kernel of the stream may start now.
template <bool PAYLOAD, bool PHASED>
__global__ void __launch_bounds__(kPermuteBlock) permute_kernel(
    const float4 *o_in, const float4 *d_in, const uint32_t *p_in, const uint32_t *perm, uint32_t n, float4 *o_out,
    float4 *d_out, uint32_t *p_out, uint32_t tiles, bool early, uint32_t *err) {
    if (early) allow_dependent_launch();
    wait_for_prerequisite();
    uint32_t first = blockIdx.x * kPermuteRays;
    if (PHASED) {
        using Tile = PhaseTile<PAYLOAD>;
        const uint32_t phase = blockIdx.x / tiles;
        first = (blockIdx.x - phase * tiles) * Tile::kRays;
        const uint32_t array = PAYLOAD ? phase : phase + 1u;
        bool in_order;
        if (array == 0)
            in_order = gather_phase<Tile::PER, Tile::ROUNDS, true, PAYLOAD>(p_in, perm, n, p_out, first, err);
        else if (array == 1)
            in_order = gather_phase<Tile::PER, Tile::ROUNDS, false, PAYLOAD>(o_in, perm, n, o_out, first, err);
        else
            in_order = gather_phase<Tile::PER, Tile::ROUNDS, false, PAYLOAD>(d_in, perm, n, d_out, first, err);
        if (!in_order) return;
        first += phase * kPermuteRays;
    }
    const uint32_t base = first + threadIdx.x;
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

// From this many rays on (75 MB of sources, and as much of results) the phases
// pay.  us with payload, buffers used in turn, all arrays at once / phases:
// random order 2.1M rays 43.4 / 42.2, 3.0M 78.5 / 58.9, 4.1M 129 / 85, 8.3M 354 /
// 241; pixel-ordered rays by a direction-first key 40.6 / 40.1, 70.2 / 55.1, 113 /
// 78, 309 / 212, by a Two Point key 36.5 / 37.4, 51.0 / 51.2, 69.0 / 68.6, 151 / 141;
// rays in order already 24.9 / 26.6, 34.9 / 37.1, 46.7 / 49.9, 91.6 / 97.8 (with no
// question for them 27.6, 38.1, 51.9, 103.7); shuffled within 65,536 rays 35.2 /
// 37.6, 48.8 / 51.7, 64.8 / 69.1, 125 / 135.
constexpr uint32_t kPhasedRays = 1u << 21;

// Blocks that an SM holds, and blocks that leave nearly every SM free.  Only
// grids that fill the device or hardly touch it let the next kernel start early:
// beside others its blocks are placed unevenly (reorders in a row, random order,
// us a launch: 100,000 rays 7.3 -> 3.2, 300,000 7.5 -> 5.6; a bounce of 60,000 rays
// on 250,000 triangles 141 -> 131.5; the same from 600,000 rays on; a bounce of
// 4,097 rays gains 0.4 us by the early start, one of 10,000 nothing).
constexpr uint32_t kPermuteBlocksPerSm = 8, kFewPermuteBlocks = 16;

template <bool PAYLOAD>
static void launch_permute(const float4 *o_in, const float4 *d_in, const uint32_t *p_in, const uint32_t *perm, uint32_t n,
                           float4 *o_out, float4 *d_out, uint32_t *p_out, uint32_t *err, int sm_count, cudaStream_t s) {
    using Tile = PhaseTile<PAYLOAD>;
    if (n >= kPhasedRays) {
        const uint32_t tiles = (n + Tile::kRays - 1) / Tile::kRays;
        launch_dependent(permute_kernel<PAYLOAD, true>, tiles * Tile::kPhases, kPermuteBlock, 0, s, o_in, d_in, p_in, perm,
                         n, o_out, d_out, p_out, tiles, false, err);
    } else {
        const uint32_t blocks = (n + kPermuteRays - 1) / kPermuteRays;
        const bool early = blocks <= kFewPermuteBlocks || blocks >= kPermuteBlocksPerSm * (uint32_t)sm_count;
        launch_dependent(permute_kernel<PAYLOAD, false>, blocks, kPermuteBlock, 0, s, o_in, d_in, p_in, perm, n, o_out, d_out,
                         p_out, 0u, early, err);
    }
}

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
    if (payload_in)
        launch_permute<true>(oi, di, payload_in, perm, n, oo, dd, payload_out, err, ds->sm_count, s);
    else
        launch_permute<false>(oi, di, nullptr, perm, n, oo, dd, nullptr, err, ds->sm_count, s);
    note_launches(1);
    return check_launch("rr_permute");
}
