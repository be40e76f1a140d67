// Sorting keys (Section 3.1, Figure 2) and the adaptive ray-length table
// (Section 3.1.6).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>

#include "rr_batch.cuh"
#include "rr_common.cuh"
#include "rr_keymath.cuh"
#include "rr_tma.cuh"

namespace rr {

struct KeyArgs {
    uint32_t *err;  // device error word
    const float4 *o_tmin;
    const float4 *d_tmax;
    uint32_t n;
    uint32_t bits;
    float lo[3], hi[3];
    float ratio;
    const float *t_given;
    const ulonglong2 *table;  // cells {sum, count}
    void *keys;
    SortCountTarget count;    // the fused form only: where the digit counts go
};

// The key of one ray (Section 3.1): the first `bits` bits of its layout's
// string, in the frame of the quantisation box.  t_given: the GIVEN estimate;
// table: the ADAPTIVE cells.
template <int LAYOUT, int TSRC, typename KeyT>
__device__ __forceinline__ KeyT ray_key(const QuantFrame &f, float4 o, float4 d, uint32_t bits, float ratio,
                                            float t_given, const ulonglong2 *table, const uint32_t *lut) {
    uint32_t qo[3], qd[3];
    float dh[3];
    quantise_ray(f, o, d, qo, qd, dh);
    uint64_t key64;
    if (LAYOUT == RR_KEY_TWO_POINT) {
        float t;
        if (TSRC == RR_T_FIXED) {
            t = __fmul_rn(ratio, f.E);
        } else if (TSRC == RR_T_GIVEN) {
            t = t_given;
        } else {
            // mean length of the ray's cell, in units of E / 2^24
            ulonglong2 cell = __ldg(table + table_cell(qo, qd));
            if (cell.y == 0ull) {
                t = __fmul_rn(0.25f, f.E);
            } else {
                const uint32_t mean = div_floor_u64(cell.x, cell.y);
                t = __fmul_rn(__fmul_rn(__uint2float_rn(mean), 5.9604644775390625e-8f), f.E);
            }
        }
        if (!isfinite(t)) t = __fmul_rn(4.0f, f.E);
        uint32_t c[6];
        c[0] = qo[0];
        c[1] = qo[1];
        c[2] = qo[2];
        c[3] = quantise_coord(f, 0, __fadd_rn(o.x, __fmul_rn(dh[0], t)));
        c[4] = quantise_coord(f, 1, __fadd_rn(o.y, __fmul_rn(dh[1], t)));
        c[5] = quantise_coord(f, 2, __fadd_rn(o.z, __fmul_rn(dh[2], t)));
        key64 = interleave6_64_lut(c, lut);
    } else if (LAYOUT == RR_KEY_AILA || LAYOUT == RR_KEY_AILA_COMPACT) {
        uint32_t c[6] = {qo[0], qo[1], qo[2], qd[0] >> 3, qd[1] >> 3, qd[2] >> 3};
        key64 = LAYOUT == RR_KEY_AILA ? interleave6_64_lut(c, lut) : interleave_compact_64(c);
    } else if (LAYOUT == RR_KEY_ORIGIN) {
        key64 = morton3_64(qo[0], qo[1], qo[2]);
    } else if (LAYOUT == RR_KEY_REIS || LAYOUT == RR_KEY_COSTA) {
        // two prefixes of their own Morton strings; the 32-bit split of Figure 2
        // (22 + 10 and 8 + 24) scaled to `bits`
        const uint32_t db = LAYOUT == RR_KEY_REIS ? (bits * 10u) / 32u : (bits * 8u) / 32u;
        const uint32_t ob = bits - db;
        const uint64_t ko = prefix64(morton3_64(qo[0], qo[1], qo[2]), ob);
        const uint64_t kd = prefix64(morton3_64(qd[0], qd[1], qd[2]), db);
        return (KeyT)(LAYOUT == RR_KEY_REIS ? (db ? (ko << db) | kd : ko) : (ob ? (kd << ob) | ko : kd));
    } else {
        float u, v;
        octahedral(d.x, d.y, d.z, u, v);
        const uint32_t c[5] = {qo[0], qo[1], qo[2], quantise_unit(u) >> 4, quantise_unit(v) >> 4};
        key64 = interleave_octa_64(c);
    }
    // a key of at most 32 bits lies in the string's first word
    if (sizeof(KeyT) == 4) return (KeyT)((uint32_t)(key64 >> 32) >> (32 - bits));
    return (KeyT)(key64 >> (64 - bits));
}

// Persistent blocks walk over tiles of 512 rays.  Each tile's origins and
// directions arrive in shared memory by two bulk asynchronous copies completed
// on an mbarrier, issued one tile ahead into the other of two buffers, so the
// loads of the next tile overlap the key arithmetic of this one (plain loads
// one tile ahead take the same time).  One ray per thread per tile:
// quantisation, interleave, one store.
//
// What bounds it: issue and shared atomics at 8.3M rays (74% of the issue
// slots, 69% of the shared-memory pipe with the digit counting; 72 us for 332
// MB, 0.68 of the copy bandwidth), launch, tail and the blocks' count flushes
// below a million.  Clamping inside the multiply and the conversion, digits at
// fixed shifts, and only one word of the string for keys of at most 32 bits
// took 8.3M 64-bit Aila keys from 88 to 71 us; blocks of 512 instead of 256
// threads and two counts per flush atomic saved keys and sort of 300,001 64-bit
// keys 5 us and of 2.07M 32-bit keys 3.
constexpr int kKeyTile = 512;
constexpr uint32_t kCopySpinLimit = 1u << 22;  // polls of a copy's barrier before giving up

// Digit-count entries of the fused form: passes x 2^radix_bits is at most 256
// a key byte with 4- or 8-bit digits.
template <typename KeyT>
constexpr uint32_t kCountEntries = 256 * sizeof(KeyT);

// Adds a key's digit of every sort pass to the counters.  Bits above the key's
// are zero, so the last pass's digit needs no narrower mask.  8-bit digits at
// fixed shifts: a loop over passes costs three times the instructions.
template <typename KeyT>
__device__ __forceinline__ void count_digits(KeyT key, uint32_t *counts, uint32_t passes, uint32_t radix_bits) {
    if (radix_bits == 8) {
#pragma unroll
        for (uint32_t p = 0; p < sizeof(KeyT); ++p)
            if (p < passes) atomicAdd(&counts[(p << 8) + ((uint32_t)(key >> (8 * p)) & 255u)], 1u);
    } else {
        for (uint32_t p = 0; p < passes; ++p) {
            atomicAdd(&counts[(p << radix_bits) + ((uint32_t)key & ((1u << radix_bits) - 1u))], 1u);
            key >>= radix_bits;
        }
    }
}

// After a block's last key: its counts (two copies) go to the sort's digit
// counts, two neighbouring 32-bit counts per 64-bit atomic (no count passes
// 2^30), and the sort's look-back words and tile counters are cleared.
__device__ __forceinline__ void finish_counts(const uint32_t *even, const uint32_t *odd, const SortCountTarget &c) {
    const uint32_t entries = c.passes << c.radix_bits;
    for (uint32_t i = 2 * threadIdx.x; i < entries; i += 2 * blockDim.x) {
        const uint32_t c0 = even[i] + odd[i], c1 = even[i + 1] + odd[i + 1];
        if (c0 | c1) atomicAdd(reinterpret_cast<unsigned long long *>(c.hist + i), (unsigned long long)c1 << 32 | c0);
    }
    if (blockIdx.x == 0 && threadIdx.x < c.passes) c.counters[threadIdx.x] = 0u;
    for (size_t w = (size_t)blockIdx.x * blockDim.x + threadIdx.x; w < c.zero_count; w += (size_t)gridDim.x * blockDim.x)
        c.zero_words[w] = make_uint4(0u, 0u, 0u, 0u);
}

// COUNT (the fused key + sort form): each block also counts the digits of
// every sort pass of its keys (shared atomics into two copies, even and odd
// warps), adds its counts to the sort's digit counts once at the end, and
// clears the sort's look-back words and tile counters, so the separate
// counting kernel of the sort is not needed.  The counters are dynamic shared
// memory: beside the two ray buffers the 16 KB of 64-bit keys'
// 8-bit digits pass the 48 KB that static shared memory is documented to reach.
template <int LAYOUT, int TSRC, typename KeyT, bool COUNT>
__global__ void __launch_bounds__(kKeyTile, 3) key_kernel(KeyArgs a) {
    __shared__ __align__(128) float4 s_o[2][kKeyTile];
    __shared__ __align__(128) float4 s_d[2][kKeyTile];
    __shared__ __align__(8) uint64_t s_bar[2];
    extern __shared__ uint32_t s_cnt[];  // COUNT: even warps' counters, then odd warps'
    const uint32_t tid = threadIdx.x;
    const uint32_t tiles = (a.n + kKeyTile - 1) / kKeyTile;
    if (tid == 0) {
        mbar_init(&s_bar[0], 1);
        mbar_init(&s_bar[1], 1);
        mbar_init_fence();
    }
    if (COUNT)
        for (uint32_t i = tid; i < 2u * kCountEntries<KeyT>; i += kKeyTile) s_cnt[i] = 0u;
    const uint32_t *lut = block_spread6_lut();
    const QuantFrame f = block_frame(a.lo, a.hi);  // synchronises: barriers, counters and table published
    auto issue = [&](uint32_t t, uint32_t buf) {
        const uint32_t first = t * kKeyTile;
        const uint32_t bytes = min((uint32_t)kKeyTile, a.n - first) * (uint32_t)sizeof(float4);
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&s_bar[buf], 2 * bytes);
        bulk_copy_g2s(s_o[buf], a.o_tmin + first, bytes, &s_bar[buf]);
        bulk_copy_g2s(s_d[buf], a.d_tmax + first, bytes, &s_bar[buf]);
    };
    if (tid == 0 && blockIdx.x < tiles) issue(blockIdx.x, 0);
    uint32_t k = 0;
    for (uint32_t t = blockIdx.x; t < tiles; t += gridDim.x, ++k) {
        const uint32_t buf = k & 1u, parity = (k >> 1) & 1u;
        const uint32_t next = t + gridDim.x;
        if (tid == 0 && next < tiles) issue(next, buf ^ 1u);
        const bool ok = mbar_wait_bounded(&s_bar[buf], parity, kCopySpinLimit);
        if (!__syncthreads_and(ok)) {
            // give up on this launch; let the copies in flight (the late one
            // into `buf` and the one already issued for the next tile) land
            // before the block's shared memory goes away
            if (tid == 0) {
                atomicOr(a.err, RR_DEVERR_COPY_TIMEOUT);
                mbar_wait_bounded(&s_bar[buf], parity, kCopySpinLimit);
                if (next < tiles) mbar_wait_bounded(&s_bar[buf ^ 1u], ((k + 1) >> 1) & 1u, kCopySpinLimit);
            }
            break;
        }
        const uint32_t i = t * kKeyTile + tid;
        if (i < a.n) {
            const float tg = TSRC == RR_T_GIVEN ? __ldg(a.t_given + i) : 0.0f;
            const KeyT key =
                ray_key<LAYOUT, TSRC, KeyT>(f, s_o[buf][tid], s_d[buf][tid], a.bits, a.ratio, tg, a.table, lut);
            static_cast<KeyT *>(a.keys)[i] = key;
            if (COUNT) count_digits(key, s_cnt + ((tid >> 5) & 1u) * kCountEntries<KeyT>, a.count.passes, a.count.radix_bits);
        }
        __syncthreads();  // every thread is done with `buf` before it is refilled
    }
    if constexpr (COUNT) {
        __syncthreads();
        finish_counts(s_cnt, s_cnt + kCountEntries<KeyT>, a.count);
    }
}

// Batches: the key of ray i in the frame (and table) of its segment, with the
// segment number above the key's bits.  Persistent blocks count the digits of
// the sort's passes as the single-wavefront form does, so the sort needs no
// counting kernel of its own.
template <int LAYOUT, int TSRC, typename KeyT>
__global__ void __launch_bounds__(kKeyTile, 3) key_batch_kernel(const BatchScene *__restrict__ segs,
                                                               const uint32_t *__restrict__ seg_offsets,
                                                               uint32_t n_segs, const float4 *__restrict__ o_tmin,
                                                               const float4 *__restrict__ d_tmax, uint32_t n,
                                                               uint32_t bits, float ratio, KeyT *__restrict__ keys,
                                                               SortCountTarget count) {
    __shared__ uint32_t s_off[kMaxBatchSegments + 1];
    __shared__ uint32_t s_cnt[2][kCountEntries<KeyT>];
    const uint32_t *lut = block_spread6_lut();
    for (uint32_t k = threadIdx.x; k <= n_segs; k += kKeyTile) s_off[k] = seg_offsets[k];
    for (uint32_t k = threadIdx.x; k < 2u * kCountEntries<KeyT>; k += kKeyTile) (&s_cnt[0][0])[k] = 0u;
    __syncthreads();
    const uint32_t tiles = (n + kKeyTile - 1) / kKeyTile;
    for (uint32_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const uint32_t i = t * kKeyTile + threadIdx.x;
        if (i >= n) break;
        uint32_t lo = 0, hi = n_segs;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (s_off[mid] <= i)
                lo = mid;
            else
                hi = mid;
        }
        const QuantFrame f = segs[lo].frame;
        const ulonglong2 *table = reinterpret_cast<const ulonglong2 *>(segs[lo].table);
        const KeyT k =
            ray_key<LAYOUT, TSRC, KeyT>(f, __ldg(o_tmin + i), __ldg(d_tmax + i), bits, ratio, 0.0f, table, lut);
        const KeyT key = (KeyT)(((uint64_t)lo << bits) | k);
        keys[i] = key;
        count_digits(key, s_cnt[(threadIdx.x >> 5) & 1u], count.passes, count.radix_bits);
    }
    __syncthreads();
    finish_counts(s_cnt[0], s_cnt[1], count);
}

__global__ void batch_frame_kernel(BatchScene *segs, const float *boxes, uint32_t n) {
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const QuantFrame f = make_frame(boxes + 6 * k, boxes + 6 * k + 3);
    segs[k].frame = f;
    segs[k].invE = __fdiv_rn(1.0f, f.E);
}

// Dynamic shared memory of a key kernel: the counters of its COUNT form.
template <typename KeyT, bool COUNT>
constexpr uint32_t key_smem() {
    return COUNT ? 2u * (uint32_t)sizeof(uint32_t) * kCountEntries<KeyT> : 0u;
}

// Blocks of one key-kernel variant that fit on the device at once (its
// occupancy is queried once per variant, after its shared-memory limit is set).
template <int LAYOUT, int TSRC, typename KeyT, bool COUNT>
static cudaError_t key_grid(uint32_t tiles, int sm_count, uint32_t *grid) {
    static std::atomic<int> bps{0};
    int v = bps.load(std::memory_order_relaxed);
    if (v == 0) {
        const auto kernel = key_kernel<LAYOUT, TSRC, KeyT, COUNT>;
        constexpr uint32_t smem = key_smem<KeyT, COUNT>();
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kernel, kKeyTile, smem);
        if (e != cudaSuccess) return e;
        v = std::max(v, 1);
        bps.store(v, std::memory_order_relaxed);
    }
    *grid = std::max(1u, std::min(tiles, (uint32_t)(sm_count * v)));
    return cudaSuccess;
}

// An error stays the thread's last CUDA error, which the caller's check reports.
template <int LAYOUT, int TSRC, typename KeyT, bool COUNT>
static void launch_keys_k(const KeyArgs &a, int sm_count, cudaStream_t s) {
    uint32_t grid = 0;
    if (key_grid<LAYOUT, TSRC, KeyT, COUNT>((a.n + kKeyTile - 1) / kKeyTile, sm_count, &grid) != cudaSuccess) return;
    key_kernel<LAYOUT, TSRC, KeyT, COUNT><<<grid, kKeyTile, key_smem<KeyT, COUNT>(), s>>>(a);
}

template <int LAYOUT, int TSRC, bool COUNT>
static void launch_keys_t(const KeyArgs &a, bool wide, int sm_count, cudaStream_t s) {
    if (wide)
        launch_keys_k<LAYOUT, TSRC, unsigned long long, COUNT>(a, sm_count, s);
    else
        launch_keys_k<LAYOUT, TSRC, uint32_t, COUNT>(a, sm_count, s);
}

template <int LAYOUT, int TSRC>
static void launch_keys(const KeyArgs &a, bool wide, bool count, int sm_count, cudaStream_t s) {
    if (count)
        launch_keys_t<LAYOUT, TSRC, true>(a, wide, sm_count, s);
    else
        launch_keys_t<LAYOUT, TSRC, false>(a, wide, sm_count, s);
}

__global__ void table_init_kernel(ulonglong2 *cells) {
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < kTableCells) cells[i] = make_ulonglong2(4194304ull /* 0.25 * 2^24 */, 1ull);
}

// After a trace: rays that hit add their fixed-point length to their cell.
// Neighbouring lanes of a warp that share a cell combine first (a segmented
// scan over runs of equal cells, which sorted rays have), then a run's last lane
// issues the two 64-bit atomics.  What bounds it: the atomics (1.2M rays: 57 MB
// in 20 us).  Grouping all lanes of a cell by match and reduce costs a round per
// distinct cell of the warp: 1.2M sorted rays 29.6 us against 19.8, in pixel
// order 44 against 22, in random order 47 against 23.  Persistent blocks: the
// frame (divisions, a barrier) is computed once for all the rays of a block.
constexpr int kAccumulateBlock = 256;
constexpr uint32_t kAccumulateBlocksPerSm = 8;
__global__ void __launch_bounds__(kAccumulateBlock) table_accumulate_kernel(unsigned long long *cells, Box box,
                                                                            const float4 *o_tmin, const float4 *d_tmax,
                                                                            const float4 *hits, uint32_t n) {
    const QuantFrame f = block_frame(box.lo, box.hi);
    const float invE = __fdiv_rn(1.0f, f.E);
    wait_for_prerequisite();
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t tiles = (n + kAccumulateBlock - 1) / kAccumulateBlock;
    for (uint32_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const uint32_t i = t * kAccumulateBlock + threadIdx.x;
        bool valid = false;
        uint32_t cell = 0, lq = 0;
        if (i < n) {
            const float4 h = hits[i], o = o_tmin[i], d = d_tmax[i];
            if (__float_as_uint(h.w) != kMiss && isfinite(h.x)) {
                uint32_t qo[3], qd[3];
                float dh[3];
                quantise_ray(f, o, d, qo, qd, dh);
                cell = table_cell(qo, qd);
                const float len = __fmul_rn(h.x, length3(d.x, d.y, d.z));
                float x = __fmul_rn(len, invE);
                if (!(x > 0.0f)) x = 0.0f;
                if (x > 64.0f) x = 64.0f;
                lq = __float2uint_rz(__fmul_rn(x, 16777216.0f));
                valid = true;
            }
        }
        // lq below 2^31 as two halves; the count above the high halves' sum
        const uint32_t mine = valid ? cell : 0xFFFFFFFFu;
        const uint32_t before = __shfl_up_sync(0xFFFFFFFFu, mine, 1);
        const uint32_t heads = __ballot_sync(0xFFFFFFFFu, lane == 0u || before != mine);
        const uint32_t start = 31u - __clz(heads & (0xFFFFFFFFu >> (31u - lane)));
        uint32_t hi = (lq >> 16) | (1u << 24), lo = lq & 0xFFFFu;
#pragma unroll
        for (uint32_t by = 1; by < 32; by <<= 1) {
            const uint32_t h2 = __shfl_up_sync(0xFFFFFFFFu, hi, by), l2 = __shfl_up_sync(0xFFFFFFFFu, lo, by);
            if (lane >= start + by) {
                hi += h2;
                lo += l2;
            }
        }
        const bool last = lane == 31u || ((heads >> (lane + 1u)) & 1u);
        if (valid && last) {
            atomicAdd(cells + 2 * (size_t)cell, ((unsigned long long)(hi & 0xFFFFFFu) << 16) + lo);
            atomicAdd(cells + 2 * (size_t)cell + 1, (unsigned long long)(hi >> 24));
        }
        __syncwarp();
    }
}

static bool box_ok(const float lo[3], const float hi[3]) {
    for (int c = 0; c < 3; ++c)
        if (!std::isfinite(lo[c]) || !std::isfinite(hi[c]) || !(lo[c] <= hi[c])) return false;
    return true;
}

static float largest_extent_host(const Box &b) {
    float e = b.hi[0] - b.lo[0];
    for (int c = 1; c < 3; ++c) {
        float x = b.hi[c] - b.lo[c];
        if (x > e) e = x;
    }
    return e;
}

cudaError_t launch_batch_frames(BatchScene *segs, const float *boxes, uint32_t n, cudaStream_t s) {
    batch_frame_kernel<<<(n + 127) / 128, 128, 0, s>>>(segs, boxes, n);
    note_launches(1);
    return cudaGetLastError();
}

template <int LAYOUT, int TSRC, typename KeyT>
static void launch_keys_batch_k(const BatchScene *segs, const uint32_t *offs, uint32_t n_segs, const float4 *o,
                                const float4 *d, uint32_t n, uint32_t bits, float ratio, void *keys,
                                const SortCountTarget &count, int sm_count, cudaStream_t s) {
    static int bps = 0;  // as key_grid
    if (bps == 0) {
        int v = 0;
        const cudaError_t e =
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, key_batch_kernel<LAYOUT, TSRC, KeyT>, kKeyTile, 0);
        bps = (e == cudaSuccess && v > 0) ? v : 1;
    }
    const uint32_t grid = std::min((n + kKeyTile - 1) / kKeyTile, (uint32_t)(sm_count * bps));
    key_batch_kernel<LAYOUT, TSRC, KeyT>
        <<<grid, kKeyTile, 0, s>>>(segs, offs, n_segs, o, d, n, bits, ratio, static_cast<KeyT *>(keys), count);
}

rr_status launch_keys_batch(const BatchScene *segs, const uint32_t *seg_offsets, uint32_t n_segs,
                            rr_key_layout layout, rr_t_source tsrc, float ratio, uint32_t key_bits,
                            uint32_t seg_bits, const float *o_tmin, const float *d_tmax, uint32_t n, void *keys,
                            uint32_t radix_bits, void *sort_workspace, int sm_count, cudaStream_t s) {
    if (n == 0) return RR_OK;
    const bool wide = key_bits + seg_bits > 32;
    const float4 *o = reinterpret_cast<const float4 *>(o_tmin);
    const float4 *d = reinterpret_cast<const float4 *>(d_tmax);
    const SortCountTarget count = sort_count_target(n, key_bits + seg_bits, radix_bits, sort_workspace, sm_count);
    const cudaError_t e = cudaMemsetAsync(count.hist, 0, sizeof(uint32_t) * (count.passes << radix_bits), s);
    if (e != cudaSuccess) return fail_cuda(e, "rr_batch keys: memset");
#define RR_KB(L, T)                                                                                              \
    wide ? launch_keys_batch_k<L, T, unsigned long long>(segs, seg_offsets, n_segs, o, d, n, key_bits, ratio, keys, \
                                                         count, sm_count, s)                                      \
         : launch_keys_batch_k<L, T, uint32_t>(segs, seg_offsets, n_segs, o, d, n, key_bits, ratio, keys, count,    \
                                               sm_count, s)
    switch (layout) {
        case RR_KEY_AILA: RR_KB(RR_KEY_AILA, 0); break;
        case RR_KEY_AILA_COMPACT: RR_KB(RR_KEY_AILA_COMPACT, 0); break;
        case RR_KEY_ORIGIN: RR_KB(RR_KEY_ORIGIN, 0); break;
        case RR_KEY_REIS: RR_KB(RR_KEY_REIS, 0); break;
        case RR_KEY_COSTA: RR_KB(RR_KEY_COSTA, 0); break;
        case RR_KEY_OCTAHEDRON: RR_KB(RR_KEY_OCTAHEDRON, 0); break;
        default:
            if (tsrc == RR_T_ADAPTIVE)
                RR_KB(RR_KEY_TWO_POINT, RR_T_ADAPTIVE);
            else
                RR_KB(RR_KEY_TWO_POINT, RR_T_FIXED);
    }
#undef RR_KB
    note_launches(1);
    return check_launch("rr_batch keys");
}

}  // namespace rr

using namespace rr;

namespace {

// The checks of rr_compute_keys (and of the key half of rr_key_sort); fills
// the kernel arguments.  RR_OK with a->n == 0 means nothing to do.
rr_status key_setup(const char *what, const float *o_tmin, const float *d_tmax, uint32_t n, const rr_key_params *p,
                    void *keys_out, KeyArgs *a) {
    const std::string w(what);
    if (!p) return fail(RR_ERR_INVALID_ARG, w + ": params is NULL");
    if (p->layout > RR_KEY_OCTAHEDRON) return fail(RR_ERR_INVALID_ARG, w + ": bad layout");
    if (p->bits < 1 || p->bits > 64) return fail(RR_ERR_INVALID_ARG, w + ": bits not in 1..64");
    if (p->layout == RR_KEY_TWO_POINT && p->t_source > RR_T_GIVEN)
        return fail(RR_ERR_INVALID_ARG, w + ": bad t_source");
    if (!box_ok(p->aabb_lo, p->aabb_hi)) return fail(RR_ERR_INVALID_ARG, w + ": bad box");
    *a = KeyArgs{};
    if (n == 0) return RR_OK;
    if (!o_tmin || !d_tmax || !keys_out) return fail(RR_ERR_INVALID_ARG, w + ": NULL buffer");
    if (!aligned16(o_tmin) || !aligned16(d_tmax))
        return fail(RR_ERR_INVALID_ARG, w + ": rays not 16-byte aligned");
    const bool wide = p->bits > 32;
    if (!aligned(keys_out, wide ? 8 : 4)) return fail(RR_ERR_INVALID_ARG, w + ": keys misaligned");
    const size_t kbytes = (wide ? 8ull : 4ull) * n;
    if (overlaps(keys_out, kbytes, o_tmin, 16ull * n) || overlaps(keys_out, kbytes, d_tmax, 16ull * n))
        return fail(RR_ERR_INVALID_ARG, w + ": keys overlap the rays");
    if (p->layout == RR_KEY_TWO_POINT) {
        if (p->t_source == RR_T_FIXED && !std::isfinite(p->ratio))
            return fail(RR_ERR_INVALID_ARG, w + ": ratio not finite");
        if (p->t_source == RR_T_GIVEN && (!p->t_given || !aligned(p->t_given, 4)))
            return fail(RR_ERR_INVALID_ARG, w + ": t_given missing or misaligned");
        if (p->t_source == RR_T_ADAPTIVE) {
            const rr_length_table *t = p->table;
            if (!t) return fail(RR_ERR_INVALID_ARG, w + ": ADAPTIVE needs a table");
            if (std::memcmp(t->box.lo, p->aabb_lo, sizeof(float) * 3) ||
                std::memcmp(t->box.hi, p->aabb_hi, sizeof(float) * 3))
                return fail(RR_ERR_INVALID_ARG, w + ": table was created for another box");
            a->table = reinterpret_cast<const ulonglong2 *>(t->cells);
        }
    }
    a->o_tmin = reinterpret_cast<const float4 *>(o_tmin);
    a->d_tmax = reinterpret_cast<const float4 *>(d_tmax);
    a->n = n;
    a->bits = p->bits;
    for (int c = 0; c < 3; ++c) {
        a->lo[c] = p->aabb_lo[c];
        a->hi[c] = p->aabb_hi[c];
    }
    a->ratio = p->ratio;
    a->t_given = p->t_given;
    a->keys = keys_out;
    return RR_OK;
}

// Launches the key kernel of the params' layout and estimate.
void launch_layout(const rr_key_params *p, const KeyArgs &a, bool count, int sms, cudaStream_t s) {
    const bool wide = p->bits > 32;
    switch (p->layout) {
        case RR_KEY_AILA: launch_keys<RR_KEY_AILA, 0>(a, wide, count, sms, s); break;
        case RR_KEY_AILA_COMPACT: launch_keys<RR_KEY_AILA_COMPACT, 0>(a, wide, count, sms, s); break;
        case RR_KEY_ORIGIN: launch_keys<RR_KEY_ORIGIN, 0>(a, wide, count, sms, s); break;
        case RR_KEY_REIS: launch_keys<RR_KEY_REIS, 0>(a, wide, count, sms, s); break;
        case RR_KEY_COSTA: launch_keys<RR_KEY_COSTA, 0>(a, wide, count, sms, s); break;
        case RR_KEY_OCTAHEDRON: launch_keys<RR_KEY_OCTAHEDRON, 0>(a, wide, count, sms, s); break;
        default:
            if (p->t_source == RR_T_FIXED)
                launch_keys<RR_KEY_TWO_POINT, RR_T_FIXED>(a, wide, count, sms, s);
            else if (p->t_source == RR_T_GIVEN)
                launch_keys<RR_KEY_TWO_POINT, RR_T_GIVEN>(a, wide, count, sms, s);
            else
                launch_keys<RR_KEY_TWO_POINT, RR_T_ADAPTIVE>(a, wide, count, sms, s);
    }
}

}  // namespace

extern "C" rr_status rr_compute_keys(const float *o_tmin, const float *d_tmax, uint32_t n,
                                     const rr_key_params *p, void *keys_out, void *stream) {
    KeyArgs a;
    rr_status st = key_setup("rr_compute_keys", o_tmin, d_tmax, n, p, keys_out, &a);
    if (st != RR_OK || n == 0) return st;
    DeviceState *ds = device_state(&st);
    if (!ds) return st;
    cudaStream_t s = as_stream(stream);
    a.err = error_word(ds, s);
    launch_layout(p, a, false, ds->sm_count, s);
    note_launches(1);
    return check_launch("rr_compute_keys");
}

extern "C" rr_status rr_key_sort(const float *o_tmin, const float *d_tmax, uint32_t n, const rr_key_params *p,
                                 void *keys_out, uint32_t *perm_out, uint32_t radix_bits, void *workspace,
                                 size_t workspace_bytes, void *stream) {
    KeyArgs a;
    rr_status st = key_setup("rr_key_sort", o_tmin, d_tmax, n, p, keys_out, &a);
    if (st != RR_OK) return st;
    st = sort_check("rr_key_sort", keys_out, nullptr, perm_out, n, p->bits, radix_bits, workspace, workspace_bytes);
    if (st != RR_OK || n == 0) return st;
    if (overlaps(perm_out, 4ull * n, o_tmin, 16ull * n) || overlaps(perm_out, 4ull * n, d_tmax, 16ull * n) ||
        overlaps(workspace, workspace_bytes, o_tmin, 16ull * n) || overlaps(workspace, workspace_bytes, d_tmax, 16ull * n))
        return fail(RR_ERR_INVALID_ARG, "rr_key_sort: buffers overlap the rays");
    DeviceState *ds = device_state(&st);
    if (!ds) return st;
    cudaStream_t s = as_stream(stream);
    a.err = error_word(ds, s);
    a.count = sort_count_target(n, p->bits, radix_bits, workspace, ds->sm_count);
    const cudaError_t e = cudaMemsetAsync(a.count.hist, 0, sizeof(uint32_t) * (a.count.passes << radix_bits), s);
    if (e != cudaSuccess) return fail_cuda(e, "rr_key_sort: memset");
    launch_layout(p, a, true, ds->sm_count, s);
    note_launches(1);
    st = check_launch("rr_key_sort");
    if (st != RR_OK) return st;
    return sort_enqueue_passes(keys_out, nullptr, perm_out, n, p->bits, radix_bits, workspace, a.err, ds->sm_count, s);
}

extern "C" rr_status rr_length_table_create(const float lo[3], const float hi[3], rr_length_table **out,
                                            void *stream) {
    if (!out || !lo || !hi) return fail(RR_ERR_INVALID_ARG, "rr_length_table_create: NULL argument");
    *out = nullptr;
    if (!box_ok(lo, hi)) return fail(RR_ERR_INVALID_ARG, "rr_length_table_create: bad box");
    rr_status st;
    if (!device_state(&st)) return st;
    rr_length_table *t = new rr_length_table();
    cudaGetDevice(&t->device);
    for (int c = 0; c < 3; ++c) {
        t->box.lo[c] = lo[c];
        t->box.hi[c] = hi[c];
    }
    t->E = largest_extent_host(t->box);
    if (!(t->E > 0.0f)) {
        delete t;
        return fail(RR_ERR_INVALID_ARG, "rr_length_table_create: box has zero extent");
    }
    cudaError_t e = lib_malloc(reinterpret_cast<void **>(&t->cells), sizeof(unsigned long long) * 2 * kTableCells);
    if (e != cudaSuccess) {
        delete t;
        cudaGetLastError();
        return fail(RR_ERR_OOM, "rr_length_table_create: cudaMalloc failed");
    }
    *out = t;
    return rr_length_table_reset(t, stream);
}

extern "C" rr_status rr_length_table_reset(rr_length_table *t, void *stream) {
    if (!t) return fail(RR_ERR_INVALID_ARG, "rr_length_table_reset: NULL table");
    table_init_kernel<<<kTableCells / 256, 256, 0, as_stream(stream)>>>(reinterpret_cast<ulonglong2 *>(t->cells));
    note_launches(1);
    return check_launch("rr_length_table_reset");
}

extern "C" rr_status rr_length_table_accumulate(rr_length_table *t, const float *o_tmin, const float *d_tmax,
                                                const float *hits, uint32_t n, void *stream) {
    if (!t) return fail(RR_ERR_INVALID_ARG, "rr_length_table_accumulate: NULL table");
    if (n == 0) return RR_OK;
    if (!o_tmin || !d_tmax || !hits) return fail(RR_ERR_INVALID_ARG, "rr_length_table_accumulate: NULL buffer");
    if (!aligned16(o_tmin) || !aligned16(d_tmax) || !aligned16(hits))
        return fail(RR_ERR_INVALID_ARG, "rr_length_table_accumulate: buffers not 16-byte aligned");
    rr_status st;
    DeviceState *ds = device_state(&st);
    if (!ds) return st;
    const uint32_t tiles = (n + kAccumulateBlock - 1) / kAccumulateBlock;
    launch_dependent(table_accumulate_kernel, std::min(tiles, kAccumulateBlocksPerSm * (uint32_t)ds->sm_count),
                     kAccumulateBlock, 0, as_stream(stream), t->cells, t->box, reinterpret_cast<const float4 *>(o_tmin),
                     reinterpret_cast<const float4 *>(d_tmax), reinterpret_cast<const float4 *>(hits), n);
    note_launches(1);
    return check_launch("rr_length_table_accumulate");
}

extern "C" rr_status rr_length_table_read(const rr_length_table *t, uint64_t *sum_host, uint32_t *cnt_host) {
    if (!t || !sum_host || !cnt_host) return fail(RR_ERR_INVALID_ARG, "rr_length_table_read: NULL argument");
    unsigned long long *tmp = new (std::nothrow) unsigned long long[2 * (size_t)kTableCells];
    if (!tmp) return fail(RR_ERR_OOM, "rr_length_table_read: host allocation failed");
    cudaError_t e = cudaMemcpy(tmp, t->cells, sizeof(unsigned long long) * 2 * kTableCells, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) {
        delete[] tmp;
        return fail_cuda(e, "rr_length_table_read");
    }
    for (uint32_t i = 0; i < kTableCells; ++i) {
        sum_host[i] = tmp[2 * (size_t)i];
        cnt_host[i] = (uint32_t)tmp[2 * (size_t)i + 1];
    }
    delete[] tmp;
    return RR_OK;
}

extern "C" rr_status rr_length_table_write(rr_length_table *t, const uint64_t *sum_host, const uint32_t *cnt_host) {
    if (!t || !sum_host || !cnt_host) return fail(RR_ERR_INVALID_ARG, "rr_length_table_write: NULL argument");
    unsigned long long *tmp = new (std::nothrow) unsigned long long[2 * (size_t)kTableCells];
    if (!tmp) return fail(RR_ERR_OOM, "rr_length_table_write: host allocation failed");
    for (uint32_t i = 0; i < kTableCells; ++i) {
        tmp[2 * (size_t)i] = sum_host[i];
        tmp[2 * (size_t)i + 1] = cnt_host[i];
    }
    cudaError_t e = cudaMemcpy(t->cells, tmp, sizeof(unsigned long long) * 2 * kTableCells, cudaMemcpyHostToDevice);
    delete[] tmp;
    if (e != cudaSuccess) return fail_cuda(e, "rr_length_table_write");
    return RR_OK;
}

extern "C" rr_status rr_length_table_destroy(rr_length_table *t) {
    if (!t) return RR_OK;
    cudaFree(t->cells);
    delete t;
    return RR_OK;
}
