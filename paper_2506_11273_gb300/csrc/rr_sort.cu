// Stable LSD radix sort of (key, index) pairs (Section 3.2), onesweep style:
// one upfront pass counts the digits of every pass; then each digit pass is a
// single kernel in which a tile counts its digits and publishes the counts,
// ranks its keys (peer masks from warp votes), resolves its global offsets by
// a decoupled look-back over the preceding tiles (pointer jumping over
// published spans), and scatters through shared memory so that global writes
// come out in runs.  Consecutive passes overlap launch and drain
// (programmatic dependent launch).
//
// What bounds it: up to one wave of tiles the latency of a tile (time stamps in
// the kernel, 1.2M 64-bit keys, us: loads 0.9, counts 1.0, ranking 2.3, scans
// 1.0, look-back 1.7, shared scatter 1.8, writes 1.3, kernel boundary 1.2),
// beyond that issue and latency together.  Hence tiles as small as one wave
// allows (plan_sort), both scans behind one barrier, and 32-bit passes once a
// 64-bit key's low half is used up.  Keys and sort together (rr_key_sort, Two Point
// keys), with the passes before these and now: 4,097 32-bit keys 29.6 -> 24.7 us,
// 65,536 64-bit 67 -> 48, 300,001 64-bit 83.5 -> 69.6, 689,149 32-bit 61 -> 50, 1.2M
// 64-bit 131 -> 121, 2.07M 32-bit 106 -> 88, 8.3M 64-bit 629 -> 558.
#include <algorithm>
#include <mutex>

#include "rr_batch.cuh"
#include "rr_common.cuh"

namespace rr {

// Look-back word of (tile t, digit d): ready bit | first tile s of the span it
// covers | count of digit d in tiles s..t.  A span starting at tile 0 is the
// inclusive prefix.
constexpr unsigned long long kReady = 1ull << 63;
constexpr uint32_t kSpinLimit = 1u << 20;   // bounded wait on a predecessor's word
constexpr int kSortBlock = 256;
constexpr int kSortWarps = kSortBlock / 32;

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(unsigned long long *p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long lookback_word(uint32_t start, uint32_t count) {
    return kReady | ((unsigned long long)start << 32) | count;
}
__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Keys per thread of a full-size tile.
template <typename K>
struct SortTile {
    static constexpr int kItems = sizeof(K) == 8 ? 12 : 16;
};

// Look-back words: 64 bits, or 32 bits for sorts of fewer than 2^20 keys in at
// most 2^11 tiles.
template <typename W>
struct LookbackWord;
template <>
struct LookbackWord<unsigned long long> {
    using W = unsigned long long;
    static __device__ __forceinline__ W load(const W *p) { return ld_relaxed(p); }
    static __device__ __forceinline__ void store(W *p, W v) { st_relaxed(p, v); }
    static __device__ __forceinline__ W make(uint32_t start, uint32_t count) { return lookback_word(start, count); }
    static __device__ __forceinline__ bool ready(W w) { return (w & kReady) != 0; }
    static __device__ __forceinline__ uint32_t start(W w) { return (uint32_t)(w >> 32) & 0x7FFFFFFFu; }
    static __device__ __forceinline__ uint32_t count(W w) { return (uint32_t)w; }
};
constexpr uint32_t kSmallSortKeys = 1u << 20;
template <>
struct LookbackWord<uint32_t> {
    using W = uint32_t;
    static __device__ __forceinline__ W load(const W *p) {
        W v;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        return v;
    }
    static __device__ __forceinline__ void store(W *p, W v) {
        asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
    }
    static __device__ __forceinline__ W make(uint32_t start, uint32_t count) { return 0x80000000u | start << 20 | count; }
    static __device__ __forceinline__ bool ready(W w) { return (w >> 31) != 0; }
    static __device__ __forceinline__ uint32_t start(W w) { return (w >> 20) & 0x7FFu; }
    static __device__ __forceinline__ uint32_t count(W w) { return w & 0xFFFFFu; }
};

template <typename K>
__device__ __forceinline__ uint32_t digit_of(K k, uint32_t shift, uint32_t mask) {
    return (uint32_t)(k >> shift) & mask;
}

// Lanes of `among` whose digit equals this lane's digit: one warp vote per
// digit bit (votes are cheap; a match instruction per key is not).  Every lane
// of the warp must call it; lanes outside `among` get an unspecified result.
template <int RBITS>
__device__ __forceinline__ uint32_t digit_peers(uint32_t dg, uint32_t among) {
    uint32_t peers = among;
#pragma unroll
    for (int b = 0; b < RBITS; ++b) {
        const uint32_t bit = (dg >> b) & 1u;
        const uint32_t vote = __ballot_sync(0xFFFFFFFFu, bit);
        peers &= bit ? vote : ~vote;
    }
    return peers;
}

// Exclusive scans of COUNT values per thread over the first `RADIX` threads
// (threads beyond contribute zero), together: one barrier.  Called by every
// thread of the block.  s_warp: COUNT * kSortWarps words, 16-byte aligned, not
// used by another scan of the block since the last barrier.
template <int RADIX, int COUNT>
__device__ __forceinline__ void scan_digits(uint32_t (&v)[COUNT], uint32_t *s_warp) {
    static_assert(kSortWarps == 8, "two 16-byte reads cover the warp totals");
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint32_t x[COUNT];
#pragma unroll
    for (int q = 0; q < COUNT; ++q) x[q] = v[q];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
        for (int q = 0; q < COUNT; ++q) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x[q], o);
            if (lane >= (uint32_t)o) x[q] += y;
        }
    }
    if (RADIX > 32) {
        if (lane == 31) {
#pragma unroll
            for (int q = 0; q < COUNT; ++q) s_warp[q * kSortWarps + warp] = x[q];
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < COUNT; ++q) {
            const uint4 a = *reinterpret_cast<const uint4 *>(s_warp + q * kSortWarps),
                        b = *reinterpret_cast<const uint4 *>(s_warp + q * kSortWarps + 4);
            x[q] += (warp > 0 ? a.x : 0u) + (warp > 1 ? a.y : 0u) + (warp > 2 ? a.z : 0u) + (warp > 3 ? a.w : 0u) +
                    (warp > 4 ? b.x : 0u) + (warp > 5 ? b.y : 0u) + (warp > 6 ? b.z : 0u);
        }
    }
#pragma unroll
    for (int q = 0; q < COUNT; ++q) v[q] = x[q] - v[q];
}

// ------------------------------------------------------------------ upfront histograms

// Counts the digits of every pass over all keys.  Plain shared atomics into
// two copies of the block's counters (even and odd warps): one atomic per key
// and pass, far fewer instructions than building warp peer masks.
template <typename K, int RBITS>
__global__ void __launch_bounds__(kSortBlock) sort_histogram_kernel(const K *__restrict__ keys, uint32_t n,
                                                                   uint32_t bits, uint32_t passes,
                                                                   uint32_t *__restrict__ hist,
                                                                   uint4 *__restrict__ zero_words,
                                                                   size_t zero_count, uint32_t *counters,
                                                                   uint32_t *zero_err) {
    constexpr int RADIX = 1 << RBITS;
    constexpr int PMAX = (64 + RBITS - 1) / RBITS;
    constexpr int KPT = 4;  // keys per thread per round
    __shared__ uint32_t sh[2][PMAX * RADIX];
    allow_dependent_launch();
    for (uint32_t i = threadIdx.x; i < 2 * PMAX * RADIX; i += kSortBlock) (&sh[0][0])[i] = 0;
    if (blockIdx.x == 0) {
        if (threadIdx.x < passes) counters[threadIdx.x] = 0u;  // tile counters of every pass
        if (threadIdx.x == 0 && zero_err) *zero_err = 0u;
    }
    __syncthreads();
    uint32_t *mine = sh[(threadIdx.x >> 5) & 1u];
    const uint32_t stride = gridDim.x * kSortBlock * KPT;
    for (uint32_t base = blockIdx.x * kSortBlock * KPT + threadIdx.x; base < n; base += stride) {
        K k[KPT];
#pragma unroll
        for (int q = 0; q < KPT; ++q) {
            const uint32_t i = base + q * kSortBlock;
            k[q] = i < n ? keys[i] : (K)0;
        }
#pragma unroll
        for (int q = 0; q < KPT; ++q) {
            if (base + q * kSortBlock < n) {
                K x = k[q];
                uint32_t left = bits;
                for (uint32_t p = 0; p < passes; ++p) {
                    const uint32_t nb = min((uint32_t)RBITS, left);
                    atomicAdd(&mine[p * RADIX + ((uint32_t)x & ((1u << nb) - 1u))], 1u);
                    x >>= RBITS;
                    left -= nb;
                }
            }
        }
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < passes * RADIX; i += kSortBlock) {
        const uint32_t c = sh[0][i] + sh[1][i];
        if (c) atomicAdd(&hist[i], c);
    }
    // the look-back words of every pass start at zero
    for (size_t i = (size_t)blockIdx.x * kSortBlock + threadIdx.x; i < zero_count; i += (size_t)gridDim.x * kSortBlock)
        zero_words[i] = make_uint4(0u, 0u, 0u, 0u);
}

// ------------------------------------------------------------------ one digit pass

template <typename K>
struct PassArgs {
    const K *keys_in;
    const uint32_t *vals_in;  // null on the first pass: the value is the input index
    K *keys_out;              // null: keys are not written
    uint32_t *high_out;       // 64-bit keys, keys_out null: the keys' high halves are written here (null: nothing)
    uint32_t *vals_out;
    uint32_t n;
    uint32_t shift;
    uint32_t mask;
    const uint32_t *hist;     // RADIX counts of this pass's digit over all keys
    void *lookback;           // [tiles][RADIX] look-back words, zero at the start
    void *lookback_next;      // the words the next pass uses, cleared here (null: none, or clear already)
    uint32_t *tile_counter;
    uint32_t *err;
};

// Shared-memory layout of one digit pass.
template <typename K, int RBITS, int ITEMS>
struct PassSmem {
    static constexpr int RADIX = 1 << RBITS;
    static constexpr int TILE = kSortBlock * ITEMS;
    // keys [TILE] | values [TILE] | per-warp counters [warps][RADIX] | tile-local
    // digit starts [RADIX] | global base per digit [RADIX] | tile counts [RADIX]
    // | misc [24]: [0] tile id, [8..23] scan scratch
    static constexpr size_t bytes =
        sizeof(K) * TILE + sizeof(uint32_t) * (TILE + kSortWarps * RADIX + 3 * RADIX + 24);
};
static_assert(PassSmem<unsigned long long, 8, 12>::bytes <= 48 * 1024 && PassSmem<uint32_t, 8, 16>::bytes <= 48 * 1024,
              "a digit pass must fit the default dynamic shared-memory limit");

// One tile of a digit pass.  FULL tiles skip every bounds check; only the
// last tile of a pass can be partial.  LATE loads the values after the
// ranking (their loads then overlap the look-back), which keeps the ranking's
// registers low enough for four blocks per SM.  ONCE asks what is written of
// the keys (all, their high halves, nothing) once and not for every key.
template <typename K, int RBITS, int ITEMS, typename W, bool ONCE, bool FULL, bool LATE>
__device__ __forceinline__ void onesweep_tile(const PassArgs<K> &a, uint32_t tile, unsigned char *smem) {
    using Word = LookbackWord<W>;
    constexpr int RADIX = 1 << RBITS;
    constexpr int TILE = kSortBlock * ITEMS;
    constexpr int WTILE = 32 * ITEMS;
    K *s_keys = reinterpret_cast<K *>(smem);
    uint32_t *s_vals = reinterpret_cast<uint32_t *>(s_keys + TILE);
    uint32_t *s_wh = s_vals + TILE;                  // [warps][RADIX]: counts, then prefix over warps
    uint32_t *s_lstart = s_wh + kSortWarps * RADIX;  // tile-local start of each digit
    uint32_t *s_gbase = s_lstart + RADIX;            // global position minus tile-local position
    uint32_t *s_cnt = s_gbase + RADIX;               // the tile's count of each digit
    uint32_t *s_misc = s_cnt + RADIX;

    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t base = tile * TILE;
    const uint32_t wbase = base + warp * WTILE;
    const auto row = [&](uint32_t t) { return static_cast<W *>(a.lookback) + (size_t)t * RADIX + tid; };

    K k[ITEMS];
    uint32_t v[ITEMS], r[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t idx = wbase + j * 32 + lane;
        if (FULL || idx < a.n) {
            k[j] = a.keys_in[idx];
            if (!LATE) v[j] = a.vals_in ? a.vals_in[idx] : idx;
        } else {
            k[j] = 0;
            if (!LATE) v[j] = 0;
        }
    }
    // while the keys arrive: the pass's digit counts, and the next pass's words
    // cleared; tiles of many keys clear them later, when fewer loads wait (32-bit
    // keys beyond 1.5M 2% faster, sorts of 100,000 keys 3% slower)
    constexpr bool CLEAR_EARLY = ITEMS <= 8 || RBITS == 4;
    const auto clear_next = [&] {
        if (a.lookback_next && tid < RADIX) static_cast<W *>(a.lookback_next)[(size_t)tile * RADIX + tid] = 0;
    };
    const uint32_t total = tid < RADIX ? a.hist[tid] : 0u;
    if (CLEAR_EARLY) clear_next();
    // The tile's digit counts, published before the ranking so that later
    // tiles looking back wait on this tile's loads only, not on its ranking
    // (counts taken from the ranking instead: 1.2M 64-bit keys 0.137 -> 0.151 ms).
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
        if (FULL || wbase + j * 32 + lane < a.n) atomicAdd(&s_cnt[digit_of(k[j], a.shift, a.mask)], 1u);
    __syncthreads();
    const uint32_t cnt = tid < RADIX ? s_cnt[tid] : 0u;
    if (tid < RADIX) Word::store(row(tile), Word::make(tile, cnt));
    if (!CLEAR_EARLY) clear_next();

    // stable rank inside the warp: items in index order (j, then lane).  The
    // peer masks of every row are independent; only the per-digit counters chain.
    const uint32_t lt = lanemask_lt();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t among = FULL ? 0xFFFFFFFFu : __ballot_sync(0xFFFFFFFFu, wbase + j * 32 + lane < a.n);
        r[j] = digit_peers<RBITS>(digit_of(k[j], a.shift, a.mask), among);
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const bool valid = FULL || wbase + j * 32 + lane < a.n;
        const uint32_t dg = digit_of(k[j], a.shift, a.mask);
        const uint32_t peers = r[j];
        const uint32_t cur = valid ? s_wh[warp * RADIX + dg] : 0u;
        __syncwarp();
        if (valid && lane == 31u - __clz(peers)) s_wh[warp * RADIX + dg] = cur + __popc(peers);
        __syncwarp();
        r[j] = cur + __popc(peers & lt);
    }
    __syncthreads();
    if (LATE) {
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t idx = wbase + j * 32 + lane;
            v[j] = (FULL || idx < a.n) ? (a.vals_in ? a.vals_in[idx] : idx) : 0u;
        }
    }

    // per digit: prefix over warps; digit starts in the output and in the tile
    if (tid < RADIX) {
        uint32_t acc = 0;
#pragma unroll
        for (int w = 0; w < kSortWarps; w += 4) {
            uint32_t c[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) c[q] = s_wh[(w + q) * RADIX + tid];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                s_wh[(w + q) * RADIX + tid] = acc;
                acc += c[q];
            }
        }
    }
    uint32_t starts[2] = {total, cnt};
    scan_digits<RADIX>(starts, s_misc + 8);
    if (tid < RADIX) {
        uint32_t excl = 0;
        if (tile > 0) {
            // decoupled look-back by pointer jumping: add the span the nearest
            // uncovered predecessor has published and continue before its
            // start; republish the wider span so successors can jump over it.
            // Spans grow as tiles finish, so a tile needs few hops even when
            // every tile of the pass runs at the same time.
            uint32_t start = tile, sum = cnt, spins = 0;
            while (start > 0) {
                const W w = Word::load(row(start - 1));
                if (!Word::ready(w)) {
                    if (++spins > kSpinLimit) {
                        atomicOr(a.err, RR_DEVERR_LOOKBACK_TIMEOUT);
                        break;
                    }
                    __nanosleep(32);
                    continue;
                }
                sum += Word::count(w);
                start = Word::start(w);
                Word::store(row(tile), Word::make(start, sum));
            }
            excl = sum - cnt;
        }
        s_lstart[tid] = starts[1];
        s_gbase[tid] = starts[0] + excl - starts[1];
    }
    __syncthreads();

    // scatter into shared memory in digit order (stable)
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        if (FULL || wbase + j * 32 + lane < a.n) {
            const uint32_t dg = digit_of(k[j], a.shift, a.mask);
            const uint32_t pos = s_lstart[dg] + s_wh[warp * RADIX + dg] + r[j];
            s_keys[pos] = k[j];
            s_vals[pos] = v[j];
        }
    }
    __syncthreads();
    // global writes in tile order: runs of equal digits land contiguously
    const auto write = [&](auto &&put_key) {
        const auto put = [&](uint32_t i) {
            const K key = s_keys[i];
            const uint32_t gpos = s_gbase[digit_of(key, a.shift, a.mask)] + i;
            if (!index_ok(gpos, a.n, a.err)) return;
            put_key(gpos, key);
            a.vals_out[gpos] = s_vals[i];
        };
        if (FULL) {
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) put(j * kSortBlock + tid);
        } else {
            const uint32_t tile_n = min((uint32_t)TILE, a.n - base);
            for (uint32_t i = tid; i < tile_n; i += kSortBlock) put(i);
        }
    };
    const auto put_whole = [&](uint32_t at, K key) { a.keys_out[at] = key; };
    const auto put_high = [&](uint32_t at, K key) { a.high_out[at] = (uint32_t)((unsigned long long)key >> 32); };
    if (!ONCE) {
        write([&](uint32_t at, K key) {
            if (a.keys_out)
                put_whole(at, key);
            else if (sizeof(K) == 8 && a.high_out)
                put_high(at, key);
        });
    } else if (a.keys_out) {
        write(put_whole);
    } else if (a.high_out) {
        write(put_high);
    } else {
        write([](uint32_t, K) {});
    }
}

// MINB blocks per SM: 3 (shortest tile latency) or 4 (more tiles in flight), as
// dispatch_pass says.  Passes of four blocks and of tiles above the full size load
// the values late.
template <typename K, int RBITS, int ITEMS, typename W, int MINB, bool ONCE>
__global__ void __launch_bounds__(kSortBlock, MINB) onesweep_kernel(PassArgs<K> a) {
    using L = PassSmem<K, RBITS, ITEMS>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint32_t *s_wh = reinterpret_cast<uint32_t *>(smem_raw + sizeof(K) * L::TILE) + L::TILE;
    uint32_t *s_cnt = s_wh + kSortWarps * L::RADIX + 2 * L::RADIX;
    uint32_t *s_misc = s_cnt + L::RADIX;
    allow_dependent_launch();
    for (uint32_t i = threadIdx.x; i < kSortWarps * L::RADIX; i += kSortBlock) s_wh[i] = 0;
    for (uint32_t i = threadIdx.x; i < (uint32_t)L::RADIX; i += kSortBlock) s_cnt[i] = 0;
    wait_for_prerequisite();
    if (threadIdx.x == 0) s_misc[0] = atomicAdd(a.tile_counter, 1u);
    __syncthreads();
    const uint32_t tile = s_misc[0];
    if ((tile + 1) * (uint32_t)L::TILE <= a.n)
        onesweep_tile<K, RBITS, ITEMS, W, ONCE, true, (MINB > 3 || ITEMS > SortTile<K>::kItems)>(a, tile, smem_raw);
    else
        onesweep_tile<K, RBITS, ITEMS, W, ONCE, false, (MINB > 3 || ITEMS > SortTile<K>::kItems)>(a, tile, smem_raw);
}

// ------------------------------------------------------------------ local (segment) sort

// One block sorts one segment of SEG = 256 * ITEMS consecutive keys entirely in
// shared memory: an LSD pass per 8-bit digit, each ranking the keys in
// position order (warp, item, lane) with the same warp-vote peer masks as the
// global passes, then scattering them back to shared memory.  The tail segment
// is padded with all-ones keys placed after the real keys, so stability keeps
// the padding last.  perm receives global indices.
template <typename K, int ITEMS>
__global__ void __launch_bounds__(kSortBlock) segment_sort_kernel(const K *__restrict__ keys_in,
                                                                 K *__restrict__ keys_out,
                                                                 uint32_t *__restrict__ perm_out, uint32_t n,
                                                                 uint32_t bits) {
    constexpr int RBITS = 8, RADIX = 256;
    constexpr int SEG = kSortBlock * ITEMS;
    constexpr int WSEG = 32 * ITEMS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    K *s_keys = reinterpret_cast<K *>(smem_raw);
    uint32_t *s_vals = reinterpret_cast<uint32_t *>(s_keys + SEG);
    uint32_t *s_wh = s_vals + SEG;                 // [warps][RADIX]
    uint32_t *s_dstart = s_wh + kSortWarps * RADIX;  // [RADIX]
    uint32_t *s_scan = s_dstart + RADIX;           // scan scratch

    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t base = blockIdx.x * (uint32_t)SEG;
    const uint32_t m = min((uint32_t)SEG, n - base);
    const uint32_t lt = lanemask_lt();
    K k[ITEMS];
    uint32_t v[ITEMS], r[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t pos = warp * WSEG + j * 32 + lane;
        k[j] = pos < m ? keys_in[base + pos] : ~(K)0;
        v[j] = pos;
    }
    const uint32_t passes = (bits + RBITS - 1) / RBITS;
    for (uint32_t p = 0; p < passes; ++p) {
        const uint32_t shift = p * RBITS;
        const uint32_t mask = (1u << min((uint32_t)RBITS, bits - shift)) - 1u;
        for (uint32_t i = tid; i < kSortWarps * RADIX; i += kSortBlock) s_wh[i] = 0;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) r[j] = digit_peers<RBITS>(digit_of(k[j], shift, mask), 0xFFFFFFFFu);
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t dg = digit_of(k[j], shift, mask);
            const uint32_t peers = r[j];
            const uint32_t cur = s_wh[warp * RADIX + dg];
            __syncwarp();
            if (lane == 31u - __clz(peers)) s_wh[warp * RADIX + dg] = cur + __popc(peers);
            __syncwarp();
            r[j] = cur + __popc(peers & lt);
        }
        __syncthreads();
        uint32_t cnt = 0;
        if (tid < RADIX) {
            for (int w = 0; w < kSortWarps; ++w) {
                const uint32_t c = s_wh[w * RADIX + tid];
                s_wh[w * RADIX + tid] = cnt;
                cnt += c;
            }
        }
        uint32_t start[1] = {cnt};
        scan_digits<RADIX>(start, s_scan);
        if (tid < RADIX) s_dstart[tid] = start[0];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t dg = digit_of(k[j], shift, mask);
            const uint32_t pos = s_dstart[dg] + s_wh[warp * RADIX + dg] + r[j];
            s_keys[pos] = k[j];
            s_vals[pos] = v[j];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t pos = warp * WSEG + j * 32 + lane;
            k[j] = s_keys[pos];
            v[j] = s_vals[pos];
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t pos = warp * WSEG + j * 32 + lane;
        if (pos < m) {
            perm_out[base + pos] = base + v[j];
            if (keys_out) keys_out[base + pos] = k[j];
        }
    }
}

template <typename K, int ITEMS>
static size_t segment_smem() {
    return (sizeof(K) + sizeof(uint32_t)) * kSortBlock * ITEMS + sizeof(uint32_t) * (kSortWarps * 256 + 256 + 16);
}

template <typename K, int ITEMS>
static cudaError_t launch_segment_sort(const K *keys_in, K *keys_out, uint32_t *perm_out, uint32_t n, uint32_t bits,
                                       cudaStream_t s) {
    const size_t smem = segment_smem<K, ITEMS>();
    static bool configured = false;
    if (!configured) {
        const cudaError_t e = cudaFuncSetAttribute(segment_sort_kernel<K, ITEMS>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const uint32_t seg = kSortBlock * ITEMS;
    segment_sort_kernel<K, ITEMS><<<(n + seg - 1) / seg, kSortBlock, smem, s>>>(keys_in, keys_out, perm_out, n, bits);
    return cudaGetLastError();
}

template <typename K>
static cudaError_t dispatch_segment_sort(const K *ki, K *ko, uint32_t *perm, uint32_t n, uint32_t bits,
                                         uint32_t segment, cudaStream_t s) {
    switch (segment) {
        case 256: return launch_segment_sort<K, 1>(ki, ko, perm, n, bits, s);
        case 512: return launch_segment_sort<K, 2>(ki, ko, perm, n, bits, s);
        case 1024: return launch_segment_sort<K, 4>(ki, ko, perm, n, bits, s);
        case 2048: return launch_segment_sort<K, 8>(ki, ko, perm, n, bits, s);
        default: return launch_segment_sort<K, 16>(ki, ko, perm, n, bits, s);
    }
}

// ------------------------------------------------------------------ host side

constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct SortPlan {
    uint32_t passes, radix, kb;
    uint32_t items;   // keys per thread of a pass over kb-byte keys
    uint32_t tiles;   // its tiles
    uint32_t wb;      // bytes of a look-back word
    uint32_t regions; // sets of look-back words: a pass clears the set of the pass after it
    uint32_t wave, wave4; // tiles that fit on the device at three and at four blocks per SM
    size_t off_hist, off_counters, off_lookback, off_keys_a, off_keys_b, off_vals, total;
};

constexpr uint32_t full_items(uint32_t kb) {
    return kb == 8 ? SortTile<unsigned long long>::kItems : SortTile<uint32_t>::kItems;
}

// Workspace layout: digit counts [pass][radix], tile counters [pass],
// look-back words, two key buffers, one value buffer.  The look-back part has
// room for a 64-bit word per pass, full-size tile and digit; two sets of words
// are used in turn.
//
// Tile size: the time of a pass of one wave is the latency of one tile, most
// of it proportional to the keys of a thread (ranking, scatter), so the keys
// are spread over as many tiles as still run at once: 4 keys per thread, then
// 8, 12 and (32-bit keys) 16.  (64-bit words would not fit the smallest tiles
// into the workspace, hence the 32-bit ones.)  Sizes and offsets in the workspace
// do not depend on the device's SMs, only the tile size and with it the part of
// the look-back words in use.
constexpr SortPlan plan_sort(uint32_t n, uint32_t bits, uint32_t radix_bits, int sm_count) {
    SortPlan p{};
    p.passes = (bits + radix_bits - 1) / radix_bits;
    p.radix = 1u << radix_bits;
    p.kb = bits > 32 ? 8u : 4u;
    const uint32_t tile = kSortBlock * full_items(p.kb);
    const uint32_t full_tiles = (n + tile - 1) / tile;
    p.items = full_items(p.kb);
    p.tiles = full_tiles;
    p.wb = 8;
    p.regions = p.passes > 1 ? 2u : 1u;
    p.wave = 3u * (uint32_t)sm_count;
    p.wave4 = 4u * (uint32_t)sm_count;
    for (uint32_t items = 4; items < full_items(p.kb); items += 4) {
        const uint32_t wb = items < 12 ? 4u : 8u;
        const uint32_t tiles = (n + kSortBlock * items - 1) / (kSortBlock * items);
        if ((wb == 4 && n >= kSmallSortKeys) || tiles > p.wave ||
            (uint64_t)wb * p.regions * tiles > 8ull * p.passes * full_tiles)
            continue;
        p.items = items;
        p.tiles = tiles;
        p.wb = wb;
        break;
    }
    size_t off = 0;
    p.off_hist = off;
    off = align256(off + sizeof(uint32_t) * p.passes * p.radix);
    p.off_counters = off;
    off = align256(off + sizeof(uint32_t) * p.passes);
    p.off_lookback = off;
    off = align256(off + sizeof(unsigned long long) * (size_t)p.passes * full_tiles * p.radix);
    p.off_keys_a = off;
    off = align256(off + (size_t)p.kb * n);
    p.off_keys_b = off;
    off = align256(off + (size_t)p.kb * n);
    p.off_vals = off;
    off = align256(off + sizeof(uint32_t) * (size_t)n);
    p.total = off;
    return p;
}

// Fewer SMs get larger tiles in place of a second wave, in the same workspace.
static_assert(plan_sort(400000, 32, 8, 152).items == 4 && plan_sort(400000, 32, 8, 76).items == 8 &&
                  plan_sort(400000, 32, 8, 76).tiles <= 3 * 76 && plan_sort(1100000, 64, 8, 76).tiles > 3 * 76 &&
                  plan_sort(400000, 32, 8, 152).total == plan_sort(400000, 32, 8, 76).total,
              "a plan is made for the SMs of its device");

// 16-byte words of a plan's look-back words, which start at zero.
constexpr size_t lookback_uint4(const SortPlan &p) { return (size_t)p.regions * p.tiles * p.radix * p.wb / 16; }

// One digit pass, launched so that it may start while the kernel before it
// drains (programmatic dependent launch; the pass waits in the kernel).
template <typename K, int RBITS, int ITEMS, typename W, int MINB, bool ONCE = false>
static cudaError_t launch_pass(const PassArgs<K> &a, cudaStream_t s) {
    if (PassSmem<K, RBITS, ITEMS>::bytes > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(onesweep_kernel<K, RBITS, ITEMS, W, MINB, ONCE>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)PassSmem<K, RBITS, ITEMS>::bytes);
        if (e != cudaSuccess) return e;
    }
    return launch_dependent(onesweep_kernel<K, RBITS, ITEMS, W, MINB, ONCE>,
                            (a.n + kSortBlock * ITEMS - 1) / (kSortBlock * ITEMS), kSortBlock,
                            PassSmem<K, RBITS, ITEMS>::bytes, s, a);
}

// Rounds in which `tiles` tiles run on a device that holds `wave` of them; a few
// beyond a full wave start as its first ones end and cost no round.
constexpr uint32_t waves(uint32_t tiles, uint32_t wave, uint32_t spare) { return (tiles + wave - 1u - spare) / wave; }

// The pass in the plan's tile size (for 64-bit plans also the passes over the
// 32-bit high halves).  Full-size passes that fit three blocks to an SM take that
// form: its tiles are the fastest.  Beyond, larger tiles may keep the pass to one
// wave: 20 keys at three blocks for 32-bit keys (1.88M to 2.33M keys on 152 SMs;
// rr_sort of 1.9M 78.4 us against 84.4 and 85.7 at three and four blocks, of 2.07M
// 80.9 against 93.6 and 85.6), 14 keys at four blocks for 64-bit keys (1.90M to
// 2.18M; 2.16M 175 us against 189 and 184).  Else four blocks where they need
// fewer waves than three, three where they need as many (us at three / four: 32-bit
// keys 2.5M 103.5 / 95.8, 2.7M 106.6 / 112.6, 3.0M 114.1 / 120.3, 4.2M 144.7 / 141.1;
// 64-bit 1.7M 174 / 150, 2.2M 196 / 209, 3.0M 247 / 240), and from two waves of four
// on four (8.3M: 245 / 241, 600 / 577).  64-bit keys at three blocks beyond one wave
// ask once what to write (2.2M 206 -> 196 us; the other forms lose 1 to 3% by it).
// No pass has more tiles than the one before it, which clears its look-back words.
template <typename K, int RBITS>
static cudaError_t dispatch_pass(const SortPlan &pl, const PassArgs<K> &a, cudaStream_t s) {
    using W64 = unsigned long long;
    if (pl.items == 4) return launch_pass<K, RBITS, 4, uint32_t, 3>(a, s);
    if (pl.items == 8) return launch_pass<K, RBITS, 8, uint32_t, 3>(a, s);
    const auto tiles_of = [&](uint32_t items) { return (a.n + kSortBlock * items - 1) / (kSortBlock * items); };
    const auto waves3 = [&](uint32_t items) { return waves(tiles_of(items), pl.wave, pl.wave / 100u); };
    const auto waves4 = [&](uint32_t items) { return waves(tiles_of(items), pl.wave4, pl.wave4 / 50u); };
    if (waves3(12) == 1 && (sizeof(K) == 8 || pl.items == 12)) return launch_pass<K, RBITS, 12, W64, 3>(a, s);
    constexpr uint32_t FULL = SortTile<K>::kItems;
    if (waves3(FULL) == 1) return launch_pass<K, RBITS, FULL, W64, 3>(a, s);
    if constexpr (RBITS == 8) {  // (4-bit digits: not measured)
        if constexpr (sizeof(K) == 4) {
            if (tiles_of(20) <= pl.wave) return launch_pass<K, RBITS, 20, W64, 3>(a, s);
        } else {
            if (waves4(FULL) > 1 && tiles_of(14) <= pl.wave4) return launch_pass<K, RBITS, 14, W64, 4>(a, s);
        }
    }
    const bool four = waves4(FULL) < waves3(FULL) || tiles_of(FULL) >= 2u * pl.wave4;
    return four ? launch_pass<K, RBITS, FULL, W64, 4>(a, s) : launch_pass<K, RBITS, FULL, W64, 3, sizeof(K) == 8>(a, s);
}

// The counting stage of a sort: the digit counts of every pass start at zero
// (a memset) and one counting kernel fills them, clearing the look-back words
// and tile counters.  zero_err (may be null) is a device word cleared too.
template <typename K, int RBITS>
static cudaError_t enqueue_count(const SortPlan &pl, const K *keys_in, uint32_t n, uint32_t bits, unsigned char *ws,
                                 uint32_t *zero_err, int sm_count, cudaStream_t s) {
    uint32_t *hist = reinterpret_cast<uint32_t *>(ws + pl.off_hist);
    uint32_t *counters = reinterpret_cast<uint32_t *>(ws + pl.off_counters);
    cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(uint32_t) * pl.passes * pl.radix, s);
    if (e != cudaSuccess) return e;
    const uint32_t per_block = kSortBlock * 4u;
    // counting-pass grid: two blocks per SM up to ~2M keys, then one block per
    // 8 rounds of keys up to eight per SM (more blocks in flight hide the
    // loads; each block adds its counters to the global histogram once)
    const uint32_t sms = (uint32_t)sm_count;
    const uint32_t hist_blocks = std::max(
        1u, std::min({(n + per_block - 1) / per_block, std::max(2u * sms, n / (8u * per_block)), 8u * sms}));
    sort_histogram_kernel<K, RBITS><<<hist_blocks, kSortBlock, 0, s>>>(
        keys_in, n, bits, pl.passes, hist, reinterpret_cast<uint4 *>(ws + pl.off_lookback), lookback_uint4(pl), counters,
        zero_err);
    note_launches(1);
    return cudaGetLastError();
}

// The digit passes of a sort whose counting stage has run (by enqueue_count
// or fused into the key kernel): one onesweep kernel per pass.  Allocates
// nothing.  When the sorted keys are not wanted, a 64-bit sort drops the low
// halves once their digits are used up, and the passes that are left move
// 32-bit keys.
template <typename K, int RBITS>
static cudaError_t enqueue_passes(const SortPlan &pl, const K *keys_in, K *keys_out, uint32_t *perm_out,
                                  uint32_t n, uint32_t bits, unsigned char *ws, uint32_t *err,
                                  cudaStream_t s) {
    uint32_t *hist = reinterpret_cast<uint32_t *>(ws + pl.off_hist);
    uint32_t *counters = reinterpret_cast<uint32_t *>(ws + pl.off_counters);
    K *keys_a = reinterpret_cast<K *>(ws + pl.off_keys_a);
    K *keys_b = reinterpret_cast<K *>(ws + pl.off_keys_b);
    uint32_t *vals_ws = reinterpret_cast<uint32_t *>(ws + pl.off_vals);
    const size_t region = (size_t)pl.tiles * pl.radix * pl.wb;
    constexpr uint32_t kLowPasses = 32 / RBITS;  // passes over the low half of a 64-bit key
    const uint32_t drop = sizeof(K) == 8 && !keys_out && pl.passes > kLowPasses ? kLowPasses - 1 : ~0u;
    const K *kin = keys_in;
    const uint32_t *vin = nullptr;
    for (uint32_t p = 0; p < pl.passes; ++p) {
        const bool final_slot = ((pl.passes - 1 - p) & 1u) == 0;
        K *kout;
        if (p == pl.passes - 1)
            kout = keys_out;
        else
            kout = final_slot ? (keys_out ? keys_out : keys_b) : keys_a;
        uint32_t *vout = final_slot ? perm_out : vals_ws;
        const uint32_t nb = std::min<uint32_t>(RBITS, bits - p * RBITS);
        const auto fill = [&](auto &a) {
            a.vals_in = vin;
            a.vals_out = vout;
            a.n = n;
            a.mask = (1u << nb) - 1u;
            a.hist = hist + p * pl.radix;
            a.lookback = ws + pl.off_lookback + (p & 1u) * region;
            // the words of the pass before this one become the next one's
            a.lookback_next = p > 0 && p + 1 < pl.passes ? ws + pl.off_lookback + ((p + 1) & 1u) * region : nullptr;
            a.tile_counter = counters + p;
            a.err = err;
        };
        cudaError_t e;
        if (p > drop && drop != ~0u) {
            PassArgs<uint32_t> a{};
            fill(a);
            a.keys_in = reinterpret_cast<const uint32_t *>(kin);
            a.keys_out = reinterpret_cast<uint32_t *>(kout);
            a.shift = p * RBITS - 32;
            e = dispatch_pass<uint32_t, RBITS>(pl, a, s);
        } else {
            PassArgs<K> a{};
            fill(a);
            a.keys_in = kin;
            a.keys_out = p == drop ? nullptr : kout;
            a.high_out = p == drop ? reinterpret_cast<uint32_t *>(kout) : nullptr;
            a.shift = p * RBITS;
            e = dispatch_pass<K, RBITS>(pl, a, s);
        }
        if (e != cudaSuccess) return e;
        kin = kout;
        vin = vout;
    }
    note_launches(pl.passes);
    return cudaGetLastError();
}

// Enqueues the whole sort: counting stage, one kernel per digit pass.
// Allocates nothing.  zero_err (may be null) is a device word cleared
// before the passes run.
template <typename K, int RBITS>
static cudaError_t enqueue_sort(const SortPlan &pl, const K *keys_in, K *keys_out, uint32_t *perm_out,
                                uint32_t n, uint32_t bits, unsigned char *ws, uint32_t *err, uint32_t *zero_err,
                                int sm_count, cudaStream_t s) {
    const cudaError_t e = enqueue_count<K, RBITS>(pl, keys_in, n, bits, ws, zero_err, sm_count, s);
    if (e != cudaSuccess) return e;
    return enqueue_passes<K, RBITS>(pl, keys_in, keys_out, perm_out, n, bits, ws, err, s);
}

template <typename K, int RBITS>
static rr_status run_sort(const SortPlan &pl, const K *keys_in, K *keys_out, uint32_t *perm_out, uint32_t n,
                          uint32_t bits, unsigned char *ws, uint32_t *err, int sm_count, cudaStream_t s) {
    const cudaError_t e = enqueue_sort<K, RBITS>(pl, keys_in, keys_out, perm_out, n, bits, ws, err, nullptr,
                                                 sm_count, s);
    if (e != cudaSuccess) return fail_cuda(e, "rr_sort");
    if (fault_fires(Fault::Launch)) return fail(RR_ERR_CUDA, "rr_sort: injected launch failure");
    return RR_OK;
}

// The sort of rr_sort (arguments already checked).
static rr_status sort_enqueue(const void *keys_in, void *keys_out, uint32_t *perm_out, uint32_t n, uint32_t bits,
                              uint32_t radix_bits, void *workspace, uint32_t *err, int sm_count, cudaStream_t s) {
    const SortPlan pl = plan_sort(n, bits, radix_bits, sm_count);
    unsigned char *ws = static_cast<unsigned char *>(workspace);
    if (pl.kb == 4) {
        const uint32_t *ki = static_cast<const uint32_t *>(keys_in);
        uint32_t *ko = static_cast<uint32_t *>(keys_out);
        return radix_bits == 8 ? run_sort<uint32_t, 8>(pl, ki, ko, perm_out, n, bits, ws, err, sm_count, s)
                               : run_sort<uint32_t, 4>(pl, ki, ko, perm_out, n, bits, ws, err, sm_count, s);
    }
    const unsigned long long *ki = static_cast<const unsigned long long *>(keys_in);
    unsigned long long *ko = static_cast<unsigned long long *>(keys_out);
    return radix_bits == 8 ? run_sort<unsigned long long, 8>(pl, ki, ko, perm_out, n, bits, ws, err, sm_count, s)
                           : run_sort<unsigned long long, 4>(pl, ki, ko, perm_out, n, bits, ws, err, sm_count, s);
}

SortCountTarget sort_count_target(uint32_t n, uint32_t bits, uint32_t radix_bits, void *workspace, int sm_count) {
    const SortPlan pl = plan_sort(n, bits, radix_bits, sm_count);
    unsigned char *ws = static_cast<unsigned char *>(workspace);
    SortCountTarget t;
    t.hist = reinterpret_cast<uint32_t *>(ws + pl.off_hist);
    t.counters = reinterpret_cast<uint32_t *>(ws + pl.off_counters);
    t.zero_words = reinterpret_cast<uint4 *>(ws + pl.off_lookback);
    t.zero_count = lookback_uint4(pl);
    t.passes = pl.passes;
    t.radix_bits = radix_bits;
    return t;
}

rr_status sort_enqueue_passes(const void *keys_in, void *keys_out, uint32_t *perm_out, uint32_t n, uint32_t bits,
                              uint32_t radix_bits, void *workspace, uint32_t *err, int sm_count, cudaStream_t s) {
    const SortPlan pl = plan_sort(n, bits, radix_bits, sm_count);
    unsigned char *ws = static_cast<unsigned char *>(workspace);
    cudaError_t e;
    if (pl.kb == 4) {
        const uint32_t *ki = static_cast<const uint32_t *>(keys_in);
        uint32_t *ko = static_cast<uint32_t *>(keys_out);
        e = radix_bits == 8 ? enqueue_passes<uint32_t, 8>(pl, ki, ko, perm_out, n, bits, ws, err, s)
                            : enqueue_passes<uint32_t, 4>(pl, ki, ko, perm_out, n, bits, ws, err, s);
    } else {
        const unsigned long long *ki = static_cast<const unsigned long long *>(keys_in);
        unsigned long long *ko = static_cast<unsigned long long *>(keys_out);
        e = radix_bits == 8
                ? enqueue_passes<unsigned long long, 8>(pl, ki, ko, perm_out, n, bits, ws, err, s)
                : enqueue_passes<unsigned long long, 4>(pl, ki, ko, perm_out, n, bits, ws, err, s);
    }
    if (e != cudaSuccess) return fail_cuda(e, "sort passes");
    if (fault_fires(Fault::Launch)) return fail(RR_ERR_CUDA, "sort passes: injected launch failure");
    return RR_OK;
}

rr_status sort_check(const char *what, const void *keys_in, const void *keys_out, const uint32_t *perm_out,
                     uint32_t n, uint32_t bits, uint32_t radix_bits, const void *workspace,
                     size_t workspace_bytes) {
    const std::string w(what);
    if (bits < 1 || bits > 64) return fail(RR_ERR_INVALID_ARG, w + ": bits not in 1..64");
    if (radix_bits != 4 && radix_bits != 8) return fail(RR_ERR_INVALID_ARG, w + ": radix_bits must be 4 or 8");
    if (n >= (1u << 30)) return fail(RR_ERR_INVALID_ARG, w + ": n must be < 2^30");
    if (n == 0) return RR_OK;
    if (!keys_in || !perm_out || !workspace) return fail(RR_ERR_INVALID_ARG, w + ": NULL buffer");
    const SortPlan pl = plan_sort(n, bits, radix_bits, 1);  // for its sizes
    if (workspace_bytes < pl.total) return fail(RR_ERR_INVALID_ARG, w + ": workspace too small");
    if (!aligned(workspace, 256)) return fail(RR_ERR_INVALID_ARG, w + ": workspace not 256-byte aligned");
    const size_t kbytes = (size_t)pl.kb * n;
    if (!aligned(keys_in, pl.kb) || (keys_out && !aligned(keys_out, pl.kb)) || !aligned(perm_out, 4))
        return fail(RR_ERR_INVALID_ARG, w + ": misaligned buffer");
    if (overlaps(keys_in, kbytes, perm_out, 4ull * n) ||
        (keys_out && (overlaps(keys_out, kbytes, keys_in, kbytes) || overlaps(keys_out, kbytes, perm_out, 4ull * n))) ||
        overlaps(workspace, pl.total, keys_in, kbytes) || overlaps(workspace, pl.total, perm_out, 4ull * n) ||
        (keys_out && overlaps(workspace, pl.total, keys_out, kbytes)))
        return fail(RR_ERR_INVALID_ARG, w + ": buffers overlap");
    return RR_OK;
}

}  // namespace rr

using namespace rr;

extern "C" rr_status rr_sort_workspace_size(uint32_t n, uint32_t bits, uint32_t radix_bits, size_t *bytes) {
    if (!bytes) return fail(RR_ERR_INVALID_ARG, "rr_sort_workspace_size: bytes is NULL");
    if (bits < 1 || bits > 64) return fail(RR_ERR_INVALID_ARG, "rr_sort_workspace_size: bits not in 1..64");
    if (radix_bits != 4 && radix_bits != 8)
        return fail(RR_ERR_INVALID_ARG, "rr_sort_workspace_size: radix_bits must be 4 or 8");
    if (n >= (1u << 30)) return fail(RR_ERR_INVALID_ARG, "rr_sort_workspace_size: n must be < 2^30");
    *bytes = plan_sort(n, bits, radix_bits, 1).total;
    return RR_OK;
}

extern "C" rr_status rr_sort(const void *keys_in, void *keys_out, uint32_t *perm_out, uint32_t n, uint32_t bits,
                             uint32_t radix_bits, void *workspace, size_t workspace_bytes, void *stream) {
    rr_status st = sort_check("rr_sort", keys_in, keys_out, perm_out, n, bits, radix_bits, workspace, workspace_bytes);
    if (st != RR_OK || n == 0) return st;
    DeviceState *ds = device_state(&st);
    if (!ds) return st;
    cudaStream_t s = as_stream(stream);
    return sort_enqueue(keys_in, keys_out, perm_out, n, bits, radix_bits, workspace, error_word(ds, s),
                        ds->sm_count, s);
}

extern "C" rr_status rr_sort_segments(const void *keys_in, void *keys_out, uint32_t *perm_out, uint32_t n,
                                      uint32_t bits, uint32_t segment, void *stream) {
    if (bits < 1 || bits > 64) return fail(RR_ERR_INVALID_ARG, "rr_sort_segments: bits not in 1..64");
    if (segment != 256 && segment != 512 && segment != 1024 && segment != 2048 && segment != 4096)
        return fail(RR_ERR_INVALID_ARG, "rr_sort_segments: segment must be 256, 512, 1024, 2048 or 4096");
    if (n >= (1u << 30)) return fail(RR_ERR_INVALID_ARG, "rr_sort_segments: n must be < 2^30");
    if (n == 0) return RR_OK;
    if (!keys_in || !perm_out) return fail(RR_ERR_INVALID_ARG, "rr_sort_segments: NULL buffer");
    const size_t kb = bits > 32 ? 8 : 4, kbytes = kb * n;
    if (!aligned(keys_in, kb) || (keys_out && !aligned(keys_out, kb)) || !aligned(perm_out, 4))
        return fail(RR_ERR_INVALID_ARG, "rr_sort_segments: misaligned buffer");
    if (overlaps(keys_in, kbytes, perm_out, 4ull * n) ||
        (keys_out && (overlaps(keys_out, kbytes, keys_in, kbytes) || overlaps(keys_out, kbytes, perm_out, 4ull * n))))
        return fail(RR_ERR_INVALID_ARG, "rr_sort_segments: buffers overlap");
    rr_status st;
    if (!device_state(&st)) return st;
    cudaStream_t s = as_stream(stream);
    const cudaError_t e =
        kb == 4 ? dispatch_segment_sort(static_cast<const uint32_t *>(keys_in), static_cast<uint32_t *>(keys_out),
                                        perm_out, n, bits, segment, s)
                : dispatch_segment_sort(static_cast<const unsigned long long *>(keys_in),
                                        static_cast<unsigned long long *>(keys_out), perm_out, n, bits, segment, s);
    if (e != cudaSuccess) return fail_cuda(e, "rr_sort_segments");
    note_launches(1);
    return RR_OK;
}

// ------------------------------------------------------------------ failure detection self-test
//
// One digit pass over two tiles of which only the second is launched: its
// look-back waits for the first tile's word, which nothing publishes, until
// the bounded spin gives up and records RR_DEVERR_LOOKBACK_TIMEOUT.  Without
// its predecessor's counts the tile scatters below its true offsets, which
// stay inside the output (all keys are zero: digit 0, positions 0..tile-1).

extern "C" rr_status rr_selftest_lookback_timeout(void *stream) {
    rr_status st;
    DeviceState *ds = device_state(&st);
    if (!ds) return st;
    using K = uint32_t;
    constexpr uint32_t tile = kSortBlock * SortTile<K>::kItems;
    const uint32_t n = 2 * tile;
    const SortPlan pl = plan_sort(n, 8, 8, ds->sm_count);  // (its full-size tile form is run here whatever the plan prefers)
    unsigned char *ws = nullptr;
    K *keys = nullptr, *keys_out = nullptr;
    uint32_t *perm = nullptr;
    cudaError_t e = cudaMalloc(&ws, pl.total);
    if (e == cudaSuccess) e = cudaMalloc(&keys, sizeof(K) * n);
    if (e == cudaSuccess) e = cudaMalloc(&keys_out, sizeof(K) * n);
    if (e == cudaSuccess) e = cudaMalloc(&perm, sizeof(uint32_t) * n);
    cudaStream_t s = as_stream(stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws, 0, pl.total, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(keys, 0, sizeof(K) * n, s);
    const uint32_t one = 1u;  // the tile counter hands the only block tile 1
    uint32_t *counter = reinterpret_cast<uint32_t *>(ws + pl.off_counters);
    if (e == cudaSuccess) e = cudaMemcpyAsync(counter, &one, sizeof(one), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        PassArgs<K> a{};
        a.keys_in = keys;
        a.vals_in = nullptr;
        a.keys_out = keys_out;
        a.vals_out = perm;
        a.n = n;
        a.shift = 0;
        a.mask = 0xFFu;
        a.hist = reinterpret_cast<const uint32_t *>(ws + pl.off_hist);
        a.lookback = ws + pl.off_lookback;
        a.tile_counter = counter;
        a.err = error_word(ds, s);
        onesweep_kernel<K, 8, SortTile<K>::kItems, unsigned long long, 3, false>
            <<<1, kSortBlock, PassSmem<K, 8, SortTile<K>::kItems>::bytes, s>>>(a);
        note_launches(1);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(ws);
    cudaFree(keys);
    cudaFree(keys_out);
    cudaFree(perm);
    if (e != cudaSuccess) return fail_cuda(e, "rr_selftest_lookback_timeout");
    return RR_OK;
}

// ------------------------------------------------------------------ sort without allocation
//
// rr_sort_noalloc: the same sort with its scratch in a file-scope device array
// instead of a caller-supplied workspace, for callers that cannot allocate
// device memory when they sort.  Nothing here allocates: not the array (it is
// part of the loaded module), not the per-device set-up, not the launches.

namespace rr {

constexpr size_t cx_max(size_t a, size_t b) { return a > b ? a : b; }

constexpr size_t kNoAllocHeader = 256;  // device error word of this entry point
constexpr size_t kNoAllocScratchBytes =
    kNoAllocHeader + cx_max(cx_max(plan_sort(RR_SORT_NOALLOC_MAX_N, 64, 8, 1).total,
                                   plan_sort(RR_SORT_NOALLOC_MAX_N, 64, 4, 1).total),
                            cx_max(plan_sort(RR_SORT_NOALLOC_MAX_N, 32, 8, 1).total,
                                   plan_sort(RR_SORT_NOALLOC_MAX_N, 32, 4, 1).total));
static_assert(kNoAllocScratchBytes <= RR_SORT_NOALLOC_SCRATCH_BYTES, "scratch bound in rr.h is too small");

static __device__ __align__(256) unsigned char g_sort_scratch[RR_SORT_NOALLOC_SCRATCH_BYTES];

struct NoAllocDevice {
    unsigned char *scratch = nullptr;  // device address of g_sort_scratch on this device
    int sm_count = 0;
};
constexpr int kNoAllocMaxDevices = 64;
static NoAllocDevice g_noalloc_dev[kNoAllocMaxDevices];
static std::mutex g_noalloc_mutex;

// Per-device set-up, done by the first call on each device with that device
// current: look up the array's device address (host code may not use the
// symbol itself) and the SM count.
static rr_status noalloc_device(NoAllocDevice **out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return RR_ERR_CUDA;
    if (dev < 0 || dev >= kNoAllocMaxDevices) return RR_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    NoAllocDevice &d = g_noalloc_dev[dev];
    if (d.scratch == nullptr) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_sort_scratch) != cudaSuccess || p == nullptr) {
            cudaGetLastError();
            return RR_ERR_CUDA;
        }
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
            cudaGetLastError();
            return RR_ERR_CUDA;
        }
        d.sm_count = sms;
        d.scratch = static_cast<unsigned char *>(p);
    }
    *out = &d;
    return RR_OK;
}

template <typename K, int RBITS>
static rr_status launch_sort_noalloc(const SortPlan &pl, const K *keys_in, K *keys_out, uint32_t *perm_out,
                                     uint32_t n, uint32_t bits, unsigned char *scratch, int sm_count,
                                     cudaStream_t s) {
    // the array keeps the last call's contents: the counting kernel clears the
    // tile counters and the look-back words before the passes.  The error word
    // at the head of the array is not cleared: its flags stay until
    // rr_device_error reads them (take_noalloc_error).
    uint32_t *err = reinterpret_cast<uint32_t *>(scratch);
    const cudaError_t e = enqueue_sort<K, RBITS>(pl, keys_in, keys_out, perm_out, n, bits, scratch + kNoAllocHeader,
                                                 err, nullptr, sm_count, s);
    return e == cudaSuccess ? RR_OK : RR_ERR_CUDA;
}

// Reads and clears the error word of rr_sort_noalloc on the current device
// (synchronous copies of four bytes; used by rr_device_error).
uint32_t take_noalloc_error() {
    uint32_t v = 0;
    const uint32_t zero = 0;
    if (cudaMemcpyFromSymbol(&v, g_sort_scratch, sizeof(v), 0, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpyToSymbol(g_sort_scratch, &zero, sizeof(zero), 0, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return v;
}

}  // namespace rr

extern "C" rr_status rr_sort_noalloc(const void *keys_in, void *keys_out, uint32_t *perm_out, uint32_t n,
                                     uint32_t bits, uint32_t radix_bits, void *stream) {
    if (bits < 1 || bits > 64 || (radix_bits != 4 && radix_bits != 8)) return RR_ERR_INVALID_ARG;
    if (n > RR_SORT_NOALLOC_MAX_N) return RR_ERR_TOO_LARGE;
    if (n == 0) return RR_OK;
    if (!keys_in || !perm_out) return RR_ERR_INVALID_ARG;
    SortPlan pl = plan_sort(n, bits, radix_bits, 1);  // for its sizes
    if (kNoAllocHeader + pl.total > sizeof(g_sort_scratch)) return RR_ERR_TOO_LARGE;
    const size_t kbytes = (size_t)pl.kb * n;
    if (!aligned(keys_in, pl.kb) || (keys_out && !aligned(keys_out, pl.kb)) || !aligned(perm_out, 4))
        return RR_ERR_INVALID_ARG;
    if (overlaps(keys_in, kbytes, perm_out, 4ull * n) ||
        (keys_out && (overlaps(keys_out, kbytes, keys_in, kbytes) || overlaps(keys_out, kbytes, perm_out, 4ull * n))))
        return RR_ERR_INVALID_ARG;
    NoAllocDevice *d = nullptr;
    const rr_status st = noalloc_device(&d);
    if (st != RR_OK) return st;
    pl = plan_sort(n, bits, radix_bits, d->sm_count);
    cudaStream_t s = as_stream(stream);
    if (pl.kb == 4) {
        const uint32_t *ki = static_cast<const uint32_t *>(keys_in);
        uint32_t *ko = static_cast<uint32_t *>(keys_out);
        return radix_bits == 8 ? launch_sort_noalloc<uint32_t, 8>(pl, ki, ko, perm_out, n, bits, d->scratch, d->sm_count, s)
                               : launch_sort_noalloc<uint32_t, 4>(pl, ki, ko, perm_out, n, bits, d->scratch, d->sm_count, s);
    }
    const unsigned long long *ki = static_cast<const unsigned long long *>(keys_in);
    unsigned long long *ko = static_cast<unsigned long long *>(keys_out);
    return radix_bits == 8
               ? launch_sort_noalloc<unsigned long long, 8>(pl, ki, ko, perm_out, n, bits, d->scratch, d->sm_count, s)
               : launch_sort_noalloc<unsigned long long, 4>(pl, ki, ko, perm_out, n, bits, d->scratch, d->sm_count, s);
}
