// Closest-hit traversal of the compressed 8-wide BVH.
//
// Persistent warps take batches of consecutive rays from a global queue, so
// which rays share a warp is decided by the order of the ray buffer: the
// coherence that reordering is meant to create (Section 4.2 measures its
// effect on control-flow and cache efficiency).  Each thread walks the
// compressed 8-wide BVH with a stack of node groups (the hit children of a
// node that remain to be visited, in the near-to-far order given by the ray's
// direction octant).  Triangles are intersected with Moller-Trumbore in fp32
// and the winning distance is refined in compensated fp32.
//
// What bounds it: instruction issue for coherent rays, the L1 data pipe and L2
// latency for incoherent ones, and for small launches the latency of the
// longest ray.  A step of the loop therefore serves both kinds of work: a lane
// tests one pending triangle and visits one node, with room for two pending
// triangle groups, so that 25 of 32 lanes are in the node branch (20 when a
// step was either a triangle or a node; a simulation of the exact traversal on
// 150,000 random-order rays).  Nodes and triangles are read by 256-bit loads,
// two slots share a packed multiply-add, the top of the stack is in shared
// memory, and a warp whose last rays run on hands each to four lanes.
// Measured against the earlier form (one step a triangle or a node, 128-bit
// loads of 80-byte nodes, local stack), 1,168,576 triangles: 2.07M camera rays
// 0.722 -> 0.574 ms, 8.3M random-order secondary rays 3.39 -> 2.77 ms, 0.99M
// any-hit shadow rays 0.273 -> 0.230 ms.
//
// Two variants serve the reordering study: indirect access (the queue hands
// out positions of an index buffer, so sorted rays are traced without being
// gathered first, Section 4.4.1) and any-hit traversal for shadow rays (the first
// triangle found inside the interval ends the ray, Section 4).
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstring>

#include "rr_batch.cuh"
#include "rr_common.cuh"
#include "rr_keymath.cuh"
#include "rr_reciprocal.cuh"
#include "rr_trace.h"

namespace rr {

constexpr int kTraceBlock = 128;

// The BVH arrays of one scene.
struct SceneRef {
    const DevNode *nodes;
    const DevTri *tris;
    uint32_t n_nodes;
    uint32_t n_tris;
};

struct TraceArgs {
    SceneRef scene;  // single-scene kernels
    const float4 *o_tmin;
    const float4 *d_tmax;
    float4 *hits;
    const uint32_t *order;  // NULL: position k traces ray k; else ray order[k]
    uint32_t n;
    bool fills_device;  // the grid has every block that fits on the device
    uint32_t *queue;  // [0] next ray, [1] finished blocks
    uint32_t *err;
    unsigned long long *table;  // length-table cells {sum, count} (accumulating kernel only)
    float tlo[3], thi[3];       // the table's box
    // batches: ray i belongs to the segment s with seg_offsets[s] <= i < seg_offsets[s + 1]
    const BatchScene *segs;
    const uint32_t *seg_offsets;
    uint32_t n_segs;
};

// Eight 32-bit words by one 256-bit load (32-byte aligned, read-only data).
struct Words8 {
    uint32_t w[8];
};
__device__ __forceinline__ Words8 load256(const void *p) {
    Words8 r;
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]), "=r"(r.w[4]), "=r"(r.w[5]), "=r"(r.w[6]), "=r"(r.w[7])
        : "l"(p));
    return r;
}

// A ray is read once: its loads and its hit's store leave L1 to the BVH (2.07M
// camera rays 0.583 -> 0.578 ms, 8.3M random-order rays 2.79 -> 2.77; triangles
// loaded the same way lose 3% on scenes whose triangles L1 holds).  An ordinary
// load behind the kernel's wait: the kernel before may have written the rays.
__device__ __forceinline__ float4 load_once(const float4 *p) {
    float4 v;
    asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

// Error-free transformations (Knuth's TwoSum, FMA-based TwoProd).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void two_prod(float a, float b, float &p, float &e) {
    p = __fmul_rn(a, b);
    e = __fmaf_rn(a, b, -p);
}

// Distance along the ray to the plane of BVH-ordered triangle k, evaluated in
// compensated fp32: t = ((v0 - o) . n) / (d . n) with n the triangle normal
// stored as hi + lo floats and v0 - o split exactly into hi + lo.  Plain fp32
// loses relative accuracy when the hit is close to the origin compared with
// |v0 - o|; this form keeps it at a few ulps.
__device__ __forceinline__ float refine_t(const SceneRef &a, uint32_t k, float4 o, float3 d) {
    const DevTri *tp = a.tris + k;
    const float nh[3] = {__ldg(tp->nhi), __ldg(tp->nhi + 1), __ldg(tp->nhi + 2)};
    const float nl[3] = {__ldg(tp->nlo), __ldg(tp->nlo + 1), __ldg(tp->nlo + 2)};
    const float vo[3] = {__ldg(tp->v0), __ldg(tp->v0 + 1), __ldg(tp->v0 + 2)};
    const float oo[3] = {o.x, o.y, o.z}, dd[3] = {d.x, d.y, d.z};
    float num_hi = 0.0f, num_lo = 0.0f, den_hi = 0.0f, den_lo = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float w, wl, p, pe, s, se;
        two_sum(vo[c], -oo[c], w, wl);  // v0 - o exactly
        two_prod(w, nh[c], p, pe);
        two_sum(num_hi, p, s, se);
        num_hi = s;
        num_lo = __fadd_rn(num_lo, __fadd_rn(__fadd_rn(se, pe), __fmaf_rn(w, nl[c], __fmul_rn(wl, nh[c]))));
        two_prod(dd[c], nh[c], p, pe);
        two_sum(den_hi, p, s, se);
        den_hi = s;
        den_lo = __fadd_rn(den_lo, __fadd_rn(__fadd_rn(se, pe), __fmul_rn(dd[c], nl[c])));
    }
    return __fdiv_rn(__fadd_rn(num_hi, num_lo), __fadd_rn(den_hi, den_lo));
}

// Byte k of a 32-bit word as the float 2^23 + byte: one byte permute puts the
// byte in the mantissa of 2^23 (no integer-to-float conversion).
template <int K>
__device__ __forceinline__ float byte_plus_2p23(uint32_t w) {
    return __uint_as_float(__byte_perm(w, 0x4B000000u, (uint32_t)K | 0x7540u));
}

// The hit children of a node, as octant-ordered inner children, and the
// triangles of its hit leaves.  Triangle groups wait in a first-in first-out
// queue, so triangles are always tested in the order in which the traversal
// met them.
struct TriGroup {
    uint32_t base;  // the node's first triangle
    uint32_t hits;  // triangle bits still to test
    uint32_t all;   // the node's triangle bits (a bit's rank among them numbers its triangle)
};

// Traversal state of a ray.  Node groups (child base, remaining hit mask in
// the near-to-far order of the ray's direction octant | inner-child mask << 8)
// are the stack entries: one push per level descended.
struct RayState {
    float4 o;  // origin, tmin
    float idx, idy, idz;
    uint32_t negmask;
    float best;               // distance of the nearest triangle so far, or tmax
    uint32_t g_base, g_mask;  // current node group
    TriGroup t;               // the triangle group being tested
    uint32_t u_hits;          // the triangle bits of the group after it (0: none)
    int sp;
};

// The nearest triangle so far: barycentrics and BVH-ordered number (kMiss
// before the first hit).
struct Hit {
    float u, v;
    uint32_t k;
};

// Stack entries a lane keeps in shared memory; deeper ones go to local memory.
// An incoherent ray's local stack misses L1 on half of its pops, in front of
// the node load that needs the entry.
constexpr int kSharedStack = 8;

// What the node visits do not need, besides RayState: the direction (read by
// triangle tests), the hit record (written about once per ray), and base and
// bits of the second triangle group.  Three ways to keep it:
//  - one scene: the hit record in shared memory, the rest in registers: 64
//    registers a thread without spills, 32 warps per SM;
//  - several scenes in 128-thread blocks (LEAN): all of it in shared memory: 56 registers, 36 warps per SM,
//    and 1,024 registers of the SM stay free, so that the one-warp blocks of the
//    host-link copy kernel run beside a full trace;
//  - four lanes to a ray: in registers (RegisterExtra).
// The other way round each was slower: one scene at 56 registers 2.91 against
// 2.77 ms for 8.3M random-order rays and 0.602 against 0.581 ms for 2.07M camera
// rays; several scenes at 64 registers 1.244 against 1.231 ms for the 3.7M rays
// of a batch of twelve wavefronts.
template <bool MULTI, int BLOCK>
constexpr bool trace_lean() {
    return MULTI && BLOCK == 128;
}
template <bool LEAN, int BLOCK>
struct LaneMem {
    float4 hit[BLOCK];
    uint2 stack[kSharedStack * BLOCK];
    float4 d[LEAN ? BLOCK : 1];
    uint2 u[LEAN ? BLOCK : 1];
};
template <bool LEAN, int BLOCK>
struct LaneExtra {
    LaneMem<LEAN, BLOCK> &m;
    uint32_t at;  // thread of the block
    float3 dir;   // unless LEAN
    uint2 second;
    __device__ __forceinline__ void begin(float4 d) {
        if (LEAN)
            m.d[at] = d;
        else
            dir = make_float3(d.x, d.y, d.z);
        set_hit(0.0f, 0.0f, kMiss);
    }
    __device__ __forceinline__ float3 d() const {
        if (!LEAN) return dir;
        const float4 x = m.d[at];
        return make_float3(x.x, x.y, x.z);
    }
    __device__ __forceinline__ void set_hit(float u, float v, uint32_t k) {
        m.hit[at] = make_float4(u, v, __uint_as_float(k), 0.0f);
    }
    __device__ __forceinline__ Hit hit() const {
        const float4 h = m.hit[at];
        return Hit{h.x, h.y, __float_as_uint(h.z)};
    }
    __device__ __forceinline__ void set_u(uint32_t base, uint32_t all) {
        if (LEAN)
            m.u[at] = make_uint2(base, all);
        else
            second = make_uint2(base, all);
    }
    __device__ __forceinline__ uint2 u() const { return LEAN ? m.u[at] : second; }
};
// The same in registers, where four lanes share a ray.
struct RegisterExtra {
    float3 dir;
    Hit best;
    uint2 second;
    __device__ __forceinline__ void begin(float4 d) {
        dir = make_float3(d.x, d.y, d.z);
        best = Hit{0.0f, 0.0f, kMiss};
        second = make_uint2(0u, 0u);
    }
    __device__ __forceinline__ float3 d() const { return dir; }
    __device__ __forceinline__ void set_hit(float u, float v, uint32_t k) { best = Hit{u, v, k}; }
    __device__ __forceinline__ Hit hit() const { return best; }
    __device__ __forceinline__ void set_u(uint32_t base, uint32_t all) { second = make_uint2(base, all); }
    __device__ __forceinline__ uint2 u() const { return second; }
};

// Drops everything the ray still had to visit.
__device__ __forceinline__ void ray_stop(RayState &r) {
    r.g_mask = 0u;
    r.t.hits = 0u;
    r.u_hits = 0u;
    r.sp = 0;
}

// The second triangle group moves up once the first is tested.
template <typename X>
__device__ __forceinline__ void next_group(RayState &r, const X &x) {
    if (r.t.hits == 0u && r.u_hits != 0u) {
        const uint2 u = x.u();
        r.t.base = u.x;
        r.t.hits = r.u_hits;
        r.t.all = u.y;
        r.u_hits = 0u;
    }
}

template <typename X>
__device__ __forceinline__ void ray_begin(RayState &r, X &x, const SceneRef &a, float4 o, float4 d) {
    x.begin(d);
    r.o = o;
    r.idx = safe_inv(d.x);
    r.idy = safe_inv(d.y);
    r.idz = safe_inv(d.z);
    r.negmask = (r.idx < 0.0f ? 1u : 0u) | (r.idy < 0.0f ? 2u : 0u) | (r.idz < 0.0f ? 4u : 0u);
    r.best = d.w;
    // the current node group starts as a virtual group holding only the root
    r.g_base = 0u;
    r.g_mask = ((a.n_nodes > 0 && o.w <= d.w) ? 1u : 0u) | (0x100u << r.negmask);
    r.t.base = r.t.hits = r.t.all = 0u;
    r.u_hits = 0u;
    r.sp = 0;
}

// Takes the nearest child of the current node group (which holds one); what
// remains of the group is left in r.g_mask.
__device__ __forceinline__ uint32_t take_child(RayState &r) {
    const uint32_t pos = __ffs(r.g_mask) - 1u;
    r.g_mask &= r.g_mask - 1u;
    const uint32_t slot = pos ^ r.negmask;
    return r.g_base + __popc((r.g_mask >> 8) & ((1u << slot) - 1u));
}

// Tables of the node visit, in shared memory: hit masks from slot bits to octant
// positions (bit s to bit s ^ octant), and leaf masks to the nibbles of their
// slots.  The swaps and spreads they replace are ALU work, which the slab tests
// already fill (2.07M camera rays 0.605 -> 0.586 ms).
struct VisitTables {
    alignas(16) uint8_t octant[8 * 256];
    uint32_t nibbles[256];
};
constexpr VisitTables visit_tables() {
    VisitTables t{};
    for (uint32_t k = 0; k < 8 * 256; ++k) {
        uint32_t h = k & 255u;
        if (k & 256u) h = ((h & 0x55u) << 1) | ((h >> 1) & 0x55u);
        if (k & 512u) h = ((h & 0x33u) << 2) | ((h >> 2) & 0x33u);
        if (k & 1024u) h = ((h & 0x0Fu) << 4) | (h >> 4);
        t.octant[k] = (uint8_t)h;
    }
    for (uint32_t k = 0; k < 256; ++k)
        for (uint32_t s = 0; s < 8; ++s)
            if ((k >> s) & 1u) t.nibbles[k] |= 15u << (4 * s);
    return t;
}
__device__ const VisitTables g_visit_tables = visit_tables();
// Called by every thread; the caller synchronises the block afterwards.
__device__ __forceinline__ const VisitTables &block_visit_tables() {
    __shared__ VisitTables s_tables;
    for (uint32_t k = threadIdx.x; k < sizeof(VisitTables) / 16; k += blockDim.x)
        reinterpret_cast<uint4 *>(&s_tables)[k] = reinterpret_cast<const uint4 *>(&g_visit_tables)[k];
    return s_tables;
}

__device__ __forceinline__ float max3f(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Two fused multiply-adds in one instruction, each rounded as fmaf.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{\n"
        "  .reg .b64 x, y, z, w;\n"
        "  mov.b64 x, {%2, %3};\n"
        "  mov.b64 y, {%4, %5};\n"
        "  mov.b64 z, {%6, %7};\n"
        "  fma.rn.f32x2 w, x, y, z;\n"
        "  mov.b64 {%0, %1}, w;\n"
        "}\n"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}

// A node's slabs along a ray: plane q of an axis lies at t = q*b + a.  The
// byte arrives as 2^23 + q, so the offset moves into a: a' = a - 2^23*b.
// Rounding a' costs at most half a quantisation step, and every stored box is
// one step larger than the child it bounds.  n, f: near and far planes per
// axis, slots 0..3 and 4..7.
struct NodeSlabs {
    float ax, ay, az, bx, by, bz;
    uint32_t nx[2], ny[2], nz[2], fx[2], fy[2], fz[2];
};
__device__ __forceinline__ NodeSlabs node_slabs(const RayState &r, const Words8 &n0, const Words8 &n1,
                                                const Words8 &n2) {
    NodeSlabs s;
    s.bx = __uint_as_float(n0.w[4]) * r.idx;
    s.by = __uint_as_float(n0.w[5]) * r.idy;
    s.bz = __uint_as_float(n0.w[6]) * r.idz;
    s.ax = fmaf(-8388608.0f, s.bx, (__uint_as_float(n0.w[0]) - r.o.x) * r.idx);
    s.ay = fmaf(-8388608.0f, s.by, (__uint_as_float(n0.w[1]) - r.o.y) * r.idy);
    s.az = fmaf(-8388608.0f, s.bz, (__uint_as_float(n0.w[2]) - r.o.z) * r.idz);
    // for a negative direction the near plane is the box's high side
    const bool sx = r.negmask & 1u, sy = r.negmask & 2u, sz = r.negmask & 4u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        s.nx[h] = sx ? n1.w[2 + h] : n1.w[h];
        s.fx[h] = sx ? n1.w[h] : n1.w[2 + h];
        s.ny[h] = sy ? n1.w[6 + h] : n1.w[4 + h];
        s.fy[h] = sy ? n1.w[4 + h] : n1.w[6 + h];
        s.nz[h] = sz ? n2.w[2 + h] : n2.w[h];
        s.fz[h] = sz ? n2.w[h] : n2.w[2 + h];
    }
    return s;
}

// The hit slots of a visited node become the ray's current group (inner
// children) and its last pending triangle group (leaves).
template <typename X>
__device__ __forceinline__ void take_hits(RayState &r, X &x, const Words8 &n0, const Words8 &n2, uint32_t hm,
                                          const VisitTables &tables) {
    const uint32_t imask = n0.w[3] & 0xFFu, tribits = n2.w[5];
    hm &= n0.w[3] >> 8;  // used slots only
    const uint32_t hits = tables.octant[r.negmask * 256u + (hm & imask)];
    // leaves: slot bit s -> nibble s, keeping the triangles the nibble holds
    const uint32_t tris = tables.nibbles[hm & ~imask] & tribits;
    r.g_base = n0.w[7];
    r.g_mask = hits | (imask << 8);
    if (tris != 0u) {
        if (r.t.hits == 0u) {
            r.t.base = n2.w[4];
            r.t.hits = tris;
            r.t.all = tribits;
        } else {
            x.set_u(n2.w[4], tribits);
            r.u_hits = tris;
        }
    }
}

// The slots of a node whose box the ray meets within [tmin, best], two slots
// to a fused multiply-add instruction.
__device__ __forceinline__ uint32_t hit_slots(const RayState &r, const NodeSlabs &s) {
    const float tmin = r.o.w, best = r.best;
    const float2 bx = make_float2(s.bx, s.bx), by = make_float2(s.by, s.by), bz = make_float2(s.bz, s.bz);
    const float2 ax = make_float2(s.ax, s.ax), ay = make_float2(s.ay, s.ay), az = make_float2(s.az, s.az);
    uint32_t hm = 0u;
#define RR_BYTES(S, W) make_float2(byte_plus_2p23<(S) & 3>(W[(S) / 4]), byte_plus_2p23<((S) & 3) + 1>(W[(S) / 4]))
#define RR_SLOTS(S)                                                                                          \
    {                                                                                                        \
        const float2 nx = fma2(RR_BYTES(S, s.nx), bx, ax), fx = fma2(RR_BYTES(S, s.fx), bx, ax);              \
        const float2 ny = fma2(RR_BYTES(S, s.ny), by, ay), fy = fma2(RR_BYTES(S, s.fy), by, ay);              \
        const float2 nz = fma2(RR_BYTES(S, s.nz), bz, az), fz = fma2(RR_BYTES(S, s.fz), bz, az);              \
        if (max3f(nx.x, ny.x, fmaxf(nz.x, tmin)) <= min3f(fx.x, fy.x, fminf(fz.x, best))) hm |= 1u << (S);    \
        if (max3f(nx.y, ny.y, fmaxf(nz.y, tmin)) <= min3f(fx.y, fy.y, fminf(fz.y, best))) hm |= 2u << (S);    \
    }
    RR_SLOTS(0) RR_SLOTS(2) RR_SLOTS(4) RR_SLOTS(6)
#undef RR_SLOTS
#undef RR_BYTES
    return hm;
}

// Moller-Trumbore of triangle k: true (with u, v, t) for a hit with
// tmin < t < best.
__device__ __forceinline__ bool meet_triangle(const RayState &r, float3 d, const SceneRef &a, uint32_t k, float &u,
                                              float &v, float &t) {
    const DevTri *tp = a.tris + k;
    const Words8 w = load256(tp);
    const float3 v0 = make_float3(__uint_as_float(w.w[0]), __uint_as_float(w.w[1]), __uint_as_float(w.w[2]));
    const float3 e1 = make_float3(__uint_as_float(w.w[3]), __uint_as_float(w.w[4]), __uint_as_float(w.w[5]));
    const float3 e2 = make_float3(__uint_as_float(w.w[6]), __uint_as_float(w.w[7]), __ldg(&tp->e2[2]));
    const float4 o = r.o;
    const float pvx = d.y * e2.z - d.z * e2.y;
    const float pvy = d.z * e2.x - d.x * e2.z;
    const float pvz = d.x * e2.y - d.y * e2.x;
    const float det = e1.x * pvx + e1.y * pvy + e1.z * pvz;
    if (det == 0.0f) return false;
    const float inv = __frcp_rn(det);
    const float tvx = o.x - v0.x, tvy = o.y - v0.y, tvz = o.z - v0.z;
    u = (tvx * pvx + tvy * pvy + tvz * pvz) * inv;
    if (!(u >= 0.0f && u <= 1.0f)) return false;
    const float qvx = tvy * e1.z - tvz * e1.y;
    const float qvy = tvz * e1.x - tvx * e1.z;
    const float qvz = tvx * e1.y - tvy * e1.x;
    v = (d.x * qvx + d.y * qvy + d.z * qvz) * inv;
    if (!(v >= 0.0f && u + v <= 1.0f)) return false;
    t = (e2.x * qvx + e2.y * qvy + e2.z * qvz) * inv;
    return t > o.w && t < r.best;
}

// Tests the first triangle of the pending group.  ANY: a hit ends the ray.
template <bool ANY, typename X>
__device__ __forceinline__ void test_one_triangle(RayState &r, X &x, const SceneRef &a, uint32_t *err) {
    const uint32_t b = __ffs(r.t.hits) - 1u;
    r.t.hits &= r.t.hits - 1u;
    const uint32_t k = r.t.base + __popc(r.t.all & ((1u << b) - 1u));
    if (!index_ok(k, a.n_tris, err)) return;
    float u, v, t;
    if (meet_triangle(r, x.d(), a, k, u, v, t)) {
        r.best = t;
        x.set_hit(u, v, k);
        if (ANY) ray_stop(r);
    }
}

template <typename X>
__device__ __forceinline__ float4 ray_result(const RayState &r, const X &x, const SceneRef &a) {
    const Hit h = x.hit();
    if (h.k == kMiss) return make_float4(__int_as_float(0x7f800000), 0.0f, 0.0f, __uint_as_float(kMiss));
    const float tr = refine_t(a, h.k, r.o, x.d());
    const float id = __uint_as_float(__ldg(&a.tris[h.k].id));  // the triangle's number in the caller's soup
    return make_float4(isfinite(tr) ? tr : r.best, h.u, h.v, id);
}

// The length-table update of one traced ray (Section 3.1.6), the arithmetic of
// table_accumulate_kernel: a ray that hit adds trunc(clamp(t*|d|/E, 0, 64)*2^24)
// and one count to the cell of its 20-bit compacted Aila code.
__device__ __forceinline__ void accumulate_hit(unsigned long long *table, const QuantFrame &f, float invE,
                                               float4 o, float3 dir, float4 h) {
    const float4 d = make_float4(dir.x, dir.y, dir.z, 0.0f);
    if (__float_as_uint(h.w) == kMiss || !isfinite(h.x)) return;
    uint32_t qo[3], qd[3];
    float dh[3];
    quantise_ray(f, o, d, qo, qd, dh);
    const uint32_t cell = table_cell(qo, qd);
    float x = __fmul_rn(__fmul_rn(h.x, length3(d.x, d.y, d.z)), invE);
    if (!(x > 0.0f)) x = 0.0f;
    if (x > 64.0f) x = 64.0f;
    atomicAdd(table + 2 * (size_t)cell, (unsigned long long)__float2uint_rz(__fmul_rn(x, 16777216.0f)));
    atomicAdd(table + 2 * (size_t)cell + 1, 1ull);
}

// One traversal step of a warp's rays: every lane tests the first pending
// triangle of its ray and, unless two triangle groups are still waiting after
// it, visits one node (after popping the next node group when the current one
// is used up).  Returns false for a lane without a ray or whose ray is
// finished.  All lanes of the warp call it together; it brings them together
// again before the node visit, which would otherwise be issued once for the
// lanes that tested a triangle and once more for those that did not.  A stack
// that would overflow records RR_DEVERR_TRACE_STACK and ends the ray as a miss.
template <bool ANY, bool LEAN, int BLOCK>
__device__ __forceinline__ bool ray_step(RayState &r, LaneExtra<LEAN, BLOCK> &x, bool live, uint2 *l_stack,
                                         const SceneRef &sc, uint32_t *err, const VisitTables &tables) {
    uint2 *s_stack = x.m.stack + x.at;  // entries BLOCK apart
    bool more = live;
    if (live && r.t.hits != 0u) {
        test_one_triangle<ANY>(r, x, sc, err);
        next_group(r, x);
    }
    __syncwarp();
    bool visit = live && r.u_hits == 0u;
    if (visit && (r.g_mask & 0xFFu) == 0u) {
        if (r.sp == 0) {
            visit = false;
            more = r.t.hits != 0u;
        } else {
            --r.sp;
            const uint2 e = r.sp < kSharedStack ? s_stack[r.sp * BLOCK] : l_stack[r.sp - kSharedStack];
            r.g_base = e.x;
            r.g_mask = e.y;
        }
    }
    if (visit) {
        const uint32_t node = take_child(r);
        bool ok = index_ok(node, sc.n_nodes, err);
        if ((r.g_mask & 0xFFu) != 0u) {
            const uint2 e = make_uint2(r.g_base, r.g_mask);
            if (r.sp < kSharedStack) {
                s_stack[r.sp * BLOCK] = e;
            } else if (r.sp < (int)kTraceStack) {
                l_stack[r.sp - kSharedStack] = e;
            } else {
                atomicOr(err, RR_DEVERR_TRACE_STACK);
                ok = false;
            }
            ++r.sp;
        }
        if (ok) {
            const DevNode *np = sc.nodes + node;
            const Words8 n0 = load256(np), n1 = load256(&np->qlo_x), n2 = load256(&np->qlo_z);
            take_hits(r, x, n0, n2, hit_slots(r, node_slabs(r, n0, n1, n2)), tables);
        } else {
            x.set_hit(0.0f, 0.0f, kMiss);
            ray_stop(r);
        }
    }
    return more;
}

// ------------------------------------------------------------------ four lanes to a ray
//
// Where a warp has few rays, the time is the latency of its longest ray: the
// instructions of a step, at one warp's issue rate, and its loads.  Four lanes
// then share a ray: each holds the whole ray state, tests two of a node's
// eight slots and one of up to four pending triangles.  The triangles of a
// group are taken four at a time in their order, and of equal distances the
// first one wins, so the result is the one-lane traversal's.  All lanes of the
// warp run the loop together.
//
// stack: the warp's shared stack rows (row e of the block's stack lies BLOCK
// entries after row e - 1); the warp's eight rays divide the rows of its 32
// lanes, 4 * kSharedStack = 32 entries each.
static_assert(4 * kSharedStack >= (int)kTraceStack, "a ray's share of the warp's stack rows is too small");

template <int BLOCK>
__device__ __forceinline__ uint32_t quad_entry(uint32_t sp, uint32_t quad) {
    return (sp >> 2) * BLOCK + (sp & 3u) * 8u + quad;
}

// The next node group of a ray whose current one is used up; false: there is none.
template <int BLOCK>
__device__ __forceinline__ bool quad_pop(RayState &r, const uint2 *stack, uint32_t quad) {
    if (r.sp == 0) return false;
    --r.sp;
    const uint2 e = stack[quad_entry<BLOCK>(r.sp, quad)];
    r.g_base = e.x;
    r.g_mask = e.y;
    return true;
}

// Takes the nearest child of the current group and keeps the rest of the group
// on the stack; false: the ray has to end.
template <int BLOCK>
__device__ __forceinline__ bool quad_take_child(RayState &r, uint2 *stack, uint32_t quad, const SceneRef &sc, uint32_t *err,
                                                uint32_t &node) {
    node = take_child(r);
    bool ok = index_ok(node, sc.n_nodes, err);
    if ((r.g_mask & 0xFFu) != 0u) {
        if (r.sp < (int)kTraceStack) {
            stack[quad_entry<BLOCK>(r.sp, quad)] = make_uint2(r.g_base, r.g_mask);  // the four lanes store the same
        } else {
            atomicOr(err, RR_DEVERR_TRACE_STACK);
            ok = false;
        }
        ++r.sp;
    }
    return ok;
}

// The winner among the triangles that a ray's four lanes tested: the nearest
// hit (ANY: the first), the first among equals.  True if one of them was hit.
// All lanes of the warp call it; a lane without a hit has t infinite.
template <bool ANY>
__device__ __forceinline__ bool quad_winner(RayState &r, RegisterExtra &x, bool hit, float u, float v, float t, uint32_t k,
                                            uint32_t quad, uint32_t j) {
    const uint32_t hits = (__ballot_sync(0xFFFFFFFFu, hit) >> (4u * quad)) & 15u;
    if (__any_sync(0xFFFFFFFFu, hit)) {
        uint32_t win;
        if (ANY) {
            win = hits ? __ffs(hits) - 1u : 0u;
        } else {
            win = j;
            float tw = t;
#pragma unroll
            for (int by = 1; by <= 2; by <<= 1) {
                const float to = __shfl_xor_sync(0xFFFFFFFFu, tw, by);
                const uint32_t wo = __shfl_xor_sync(0xFFFFFFFFu, win, by);
                if (to < tw || (to == tw && wo < win)) {
                    tw = to;
                    win = wo;
                }
            }
        }
        const uint32_t from = 4u * quad + win;
        const float tw = __shfl_sync(0xFFFFFFFFu, t, from), uw = __shfl_sync(0xFFFFFFFFu, u, from),
                    vw = __shfl_sync(0xFFFFFFFFu, v, from);
        const uint32_t kw = __shfl_sync(0xFFFFFFFFu, k, from);
        if (hits != 0u) {
            r.best = tw;
            x.set_hit(uw, vw, kw);
            if (ANY) ray_stop(r);
        }
    }
    return hits != 0u;
}

// Whether the ray meets slot j + 4 * h of a node.
__device__ __forceinline__ bool quad_slot(const RayState &r, const NodeSlabs &s, uint32_t j, int h) {
    const uint32_t sel = 0x7540u | j;  // byte j, then the mantissa and exponent of 2^23
    const auto at = [&](uint32_t w, float b, float a) {
        return fmaf(__uint_as_float(__byte_perm(w, 0x4B000000u, sel)), b, a);
    };
    const float t0 = max3f(at(s.nx[h], s.bx, s.ax), at(s.ny[h], s.by, s.ay), fmaxf(at(s.nz[h], s.bz, s.az), r.o.w));
    const float t1 = min3f(at(s.fx[h], s.bx, s.ax), at(s.fy[h], s.by, s.ay), fminf(at(s.fz[h], s.bz, s.az), r.best));
    return t0 <= t1;
}

// The hit slots of a ray's node from those of its lanes; all lanes of the warp call it.
__device__ __forceinline__ uint32_t quad_slots(bool lo, bool hi, uint32_t quad) {
    const uint32_t l = __ballot_sync(0xFFFFFFFFu, lo), h = __ballot_sync(0xFFFFFFFFu, hi);
    return ((l >> (4u * quad)) & 15u) | (((h >> (4u * quad)) & 15u) << 4);
}

// One step: up to four pending triangles, or the next node.  Returns false
// for the lanes of a ray that is finished (or of no ray).
template <bool ANY, int BLOCK>
__device__ __forceinline__ bool quad_step(RayState &r, RegisterExtra &x, bool live, uint2 *stack, const SceneRef &sc,
                                          uint32_t *err, const VisitTables &tables) {
    const uint32_t lane = threadIdx.x & 31u, quad = lane >> 2, j = lane & 3u;
    const bool test = live && r.t.hits != 0u;
    if (__any_sync(0xFFFFFFFFu, test)) {
        float u = 0.0f, v = 0.0f, t = __int_as_float(0x7f800000);
        uint32_t k = kMiss;
        bool hit = false;
        if (test) {
            const uint32_t h0 = r.t.hits, h1 = h0 & (h0 - 1u), h2 = h1 & (h1 - 1u), h3 = h2 & (h2 - 1u);
            const uint32_t mine = j == 0u ? h0 : j == 1u ? h1 : j == 2u ? h2 : h3;
            if (mine != 0u) {
                k = r.t.base + __popc(r.t.all & ((mine & (0u - mine)) - 1u));
                if (index_ok(k, sc.n_tris, err)) hit = meet_triangle(r, x.d(), sc, k, u, v, t);
                if (!hit) t = __int_as_float(0x7f800000);
            }
            r.t.hits = h3 & (h3 - 1u);
            next_group(r, x);
        }
        quad_winner<ANY>(r, x, hit, u, v, t, k, quad, j);
    }
    __syncwarp();
    bool visit = live && r.t.hits == 0u, more = live;
    if (visit && (r.g_mask & 0xFFu) == 0u) visit = more = quad_pop<BLOCK>(r, stack, quad);
    Words8 n0{}, n2{};
    bool two[2] = {false, false};
    if (visit) {
        uint32_t node;
        visit = quad_take_child<BLOCK>(r, stack, quad, sc, err, node);
        if (visit) {
            const DevNode *np = sc.nodes + node;
            n0 = load256(np);
            n2 = load256(&np->qlo_z);
            const NodeSlabs s = node_slabs(r, n0, load256(&np->qlo_x), n2);
#pragma unroll
            for (int h = 0; h < 2; ++h) two[h] = quad_slot(r, s, j, h);
        } else {
            x.set_hit(0.0f, 0.0f, kMiss);
            ray_stop(r);
        }
    }
    const uint32_t hm = quad_slots(two[0], two[1], quad);
    if (visit) take_hits(r, x, n0, n2, hm, tables);
    return more;
}

// One step of launches of few rays: up to four pending triangles and, unless
// triangles of two groups are left after them, the next node, which is loaded
// before the triangles are tested, so that both latencies overlap (80
// registers: the tail of trace_kernel has no room for it, and the two steps
// compiled from one source disturb its main loop).  Returns as quad_step.
template <bool ANY, int BLOCK>
__device__ __forceinline__ bool quad_step_early(RayState &r, RegisterExtra &x, bool live, uint2 *stack, const SceneRef &sc,
                                                uint32_t *err, const VisitTables &tables) {
    const uint32_t lane = threadIdx.x & 31u, quad = lane >> 2, j = lane & 3u;
    // the triangles this step tests, and the node it visits
    uint32_t left = r.t.hits, mine = left;
#pragma unroll
    for (uint32_t q = 0; q < 4u; ++q) {
        if (q == j) mine = left;
        left &= left - 1u;
    }
    const bool test = live && r.t.hits != 0u;
    bool visit = live && (r.u_hits == 0u || left == 0u);
    if (visit && (r.g_mask & 0xFFu) == 0u) visit = quad_pop<BLOCK>(r, stack, quad);
    const bool more = visit || test;
    Words8 n0{}, n1{}, n2{};
    if (visit) {
        uint32_t node;
        visit = quad_take_child<BLOCK>(r, stack, quad, sc, err, node);
        if (!visit) {
            x.set_hit(0.0f, 0.0f, kMiss);
            ray_stop(r);
        } else {
            const DevNode *np = sc.nodes + node;
            n0 = load256(np);
            n1 = load256(&np->qlo_x);
            n2 = load256(&np->qlo_z);
        }
    }
    if (__any_sync(0xFFFFFFFFu, test)) {
        float u = 0.0f, v = 0.0f, t = __int_as_float(0x7f800000);
        uint32_t k = kMiss;
        bool hit = false;
        if (live && r.t.hits != 0u) {
            if (mine != 0u) {
                k = r.t.base + __popc(r.t.all & ((mine & (0u - mine)) - 1u));
                if (index_ok(k, sc.n_tris, err)) hit = meet_triangle(r, x.d(), sc, k, u, v, t);
                if (!hit) t = __int_as_float(0x7f800000);
            }
            r.t.hits = left;
            next_group(r, x);
        }
        if (quad_winner<ANY>(r, x, hit, u, v, t, k, quad, j) && ANY) visit = false;
    }
    __syncwarp();
    bool two[2] = {false, false};
    if (visit) {
        const NodeSlabs s = node_slabs(r, n0, n1, n2);
#pragma unroll
        for (int h = 0; h < 2; ++h) two[h] = quad_slot(r, s, j, h);
    }
    const uint32_t hm = quad_slots(two[0], two[1], quad);
    if (visit) take_hits(r, x, n0, n2, hm, tables);
    return more;
}

// Lanes refill from the queue once this many of a warp's 32 lanes are idle
// (their rays finished): finished lanes write their hits together and idle
// lanes take consecutive queue positions together.
constexpr uint32_t kRefillLanes = 8;

// With the queue empty, a warp left with this many rays or fewer goes on with
// four lanes to each: its longest rays decide when the launch ends (689,149
// rays through the permutation, keys and sort included: 0.396 ms without the
// hand-over, 0.362 ms with it).
constexpr uint32_t kTailRays = 8;

// Resident blocks asked of the compiler (see LaneExtra).
template <bool MULTI, int BLOCK>
constexpr int trace_min_blocks() {
    return (trace_lean<MULTI, BLOCK>() ? 1152 : 1024) / BLOCK;
}

// Dynamic shared memory of the batch kernels: the scene of every segment, then
// the segment offsets.
inline size_t multi_smem(uint32_t n_segs) { return sizeof(SceneRef) * n_segs + sizeof(uint32_t) * (n_segs + 1); }

// What the trace kernels share around the traversal.
//
// MULTI: rays of several scenes in one launch (a batch); each lane finds the
// segment of its ray when it takes the ray and traces that segment's BVH
// (and updates its table).  The segments' scenes sit in shared memory, so a
// lane keeps only its segment number in registers during traversal.
template <bool ACCUM, bool MULTI>
struct TraceContext {
    const TraceArgs &a;
    SceneRef *s_sc;
    uint32_t *s_off;
    // the table's quantisation frame is the same for the whole launch: it lives
    // in shared memory, not in every thread's registers during traversal
    QuantFrame *s_frame;
    float *s_invE;

    // Called by every thread; the caller synchronises the block afterwards.
    __device__ __forceinline__ void load() const {
        if (ACCUM && !MULTI && threadIdx.x == 0) {
            *s_frame = make_frame(a.tlo, a.thi);
            *s_invE = __fdiv_rn(1.0f, s_frame->E);
        }
        if (MULTI) {
            for (uint32_t k = threadIdx.x; k <= a.n_segs; k += blockDim.x) s_off[k] = a.seg_offsets[k];
            for (uint32_t k = threadIdx.x; k < a.n_segs; k += blockDim.x) {
                const BatchScene *bs = a.segs + k;
                s_sc[k].nodes = bs->nodes;
                s_sc[k].tris = bs->tris;
                s_sc[k].n_nodes = bs->n_nodes;
                s_sc[k].n_tris = bs->n_tris;
            }
        }
    }
    __device__ __forceinline__ const SceneRef &scene(uint32_t seg) const { return MULTI ? s_sc[seg] : a.scene; }

    // Queue position pos -> ray and segment.  false: not a position, or (an
    // index buffer that is no permutation) no ray of the launch.
    __device__ __forceinline__ bool find_ray(uint32_t pos, uint32_t &ray, uint32_t &seg) const {
        if (pos >= a.n) return false;
        const uint32_t i = a.order ? a.order[pos] : pos;
        if (i >= a.n) {  // not a permutation of [0, n): record and skip
            atomicOr(a.err, RR_DEVERR_BAD_INDEX);
            return false;
        }
        ray = i;
        if (MULTI) {
            // the last segment starting at or before i (empty segments share
            // their start with the next one, which wins)
            uint32_t lo = 0, hi = a.n_segs;
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if (s_off[mid] <= i)
                    lo = mid;
                else
                    hi = mid;
            }
            seg = lo;
        }
        return true;
    }

    template <typename X>
    __device__ __forceinline__ void store(const RayState &r, const X &x, uint32_t ray, uint32_t seg) const {
        const float4 h = ray_result(r, x, scene(seg));
        __stcs(a.hits + ray, h);
        if (ACCUM) {
            if (MULTI) {
                const BatchScene *bs = a.segs + seg;
                if (bs->table) accumulate_hit(bs->table, bs->frame, bs->invE, r.o, x.d(), h);
            } else if (a.table) {
                accumulate_hit(a.table, *s_frame, *s_invE, r.o, x.d(), h);
            }
        }
    }

    // The last block to leave the launch resets the queue for the next one.
    __device__ __forceinline__ void leave() const {
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            const uint32_t prev = atomicAdd(a.queue + 1, 1u);
            if (prev == gridDim.x - 1) {  // every block has stopped fetching
                a.queue[0] = 0u;
                a.queue[1] = 0u;
            }
        }
    }
};

// Each lane traces its own ray, at most one triangle and one node per loop
// iteration, and lanes whose ray has finished are refilled from the queue
// (kRefillLanes at a time) instead of idling until the warp's slowest ray is
// done.
template <bool ACCUM, bool ANY, bool MULTI, int BLOCK>
__global__ void __launch_bounds__(BLOCK, (trace_min_blocks<MULTI, BLOCK>())) trace_kernel(TraceArgs a) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ QuantFrame s_frame;
    __shared__ float s_invE;
    constexpr bool LEAN = trace_lean<MULTI, BLOCK>();
    __shared__ LaneMem<LEAN, BLOCK> s_lane;
    SceneRef *s_sc = reinterpret_cast<SceneRef *>(s_dyn);
    const TraceContext<ACCUM, MULTI> cx{a, s_sc, reinterpret_cast<uint32_t *>(s_sc + (MULTI ? a.n_segs : 0)), &s_frame,
                                        &s_invE};
    if (a.fills_device) allow_dependent_launch();
    const VisitTables &tables = block_visit_tables();
    wait_for_prerequisite();
    cx.load();
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t lanes_below = (1u << lane) - 1u;
    LaneExtra<LEAN, BLOCK> x{s_lane, threadIdx.x, make_float3(0.0f, 0.0f, 0.0f), make_uint2(0u, 0u)};
    uint2 l_stack[kTraceStack - kSharedStack];
    RayState r;
    uint32_t ray = 0, seg = 0;
    bool live = false, finished = false, exhausted = false;
    while (true) {
        const uint32_t idle = __ballot_sync(0xFFFFFFFFu, !live);
        if ((uint32_t)__popc(idle) >= kRefillLanes) {
            if (finished) {  // the hits of the lanes whose rays finished
                cx.store(r, x, ray, seg);
                finished = false;
            }
            if (!exhausted) {
                // idle lanes take consecutive queue positions, in lane order
                const uint32_t want = __popc(idle);
                uint32_t base = 0;
                if (lane == 0) base = atomicAdd(a.queue, want);
                base = __shfl_sync(0xFFFFFFFFu, base, 0);
                if (base + want >= a.n) exhausted = true;
                if (!live && cx.find_ray(base + __popc(idle & lanes_below), ray, seg)) {
                    ray_begin(r, x, cx.scene(seg), load_once(a.o_tmin + ray), load_once(a.d_tmax + ray));
                    live = true;
                }
            }
            if (exhausted && (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, live)) <= kTailRays) break;
        }
        const bool more = ray_step<ANY, LEAN, BLOCK>(r, x, live, l_stack, cx.scene(seg), a.err, tables);
        finished = finished || (live && !more);
        live = more;
    }
    // the tail: at most eight rays are left, four lanes take each
    const uint32_t rays = __ballot_sync(0xFFFFFFFFu, live);
    if (rays != 0u) {
        const uint32_t quad = lane >> 2;
        uint2 *stack = s_lane.stack + (threadIdx.x & ~31u);
        // owners move their stacks to their ray's rows (read before any is written)
        uint2 e[kSharedStack];
#pragma unroll
        for (int i = 0; i < kSharedStack; ++i) e[i] = s_lane.stack[i * BLOCK + threadIdx.x];
        __syncwarp();
        if (live) {
            const uint32_t to = __popc(rays & lanes_below);
#pragma unroll
            for (int i = 0; i < kSharedStack; ++i)
                if (i < r.sp) stack[quad_entry<BLOCK>(i, to)] = e[i];
            for (int i = kSharedStack; i < r.sp; ++i) stack[quad_entry<BLOCK>(i, to)] = l_stack[i - kSharedStack];
        }
        __syncwarp();
        // the lane whose ray this lane's four take over
        uint32_t left = rays;
        for (uint32_t q = 0; q < quad; ++q) left &= left - 1u;
        const uint32_t from = left ? __ffs(left) - 1u : 0u;
        RayState q;
#define RR_TAKE(F) q.F = __shfl_sync(0xFFFFFFFFu, r.F, from);
        RR_TAKE(o.x) RR_TAKE(o.y) RR_TAKE(o.z) RR_TAKE(o.w)
        RR_TAKE(idx) RR_TAKE(idy) RR_TAKE(idz) RR_TAKE(negmask) RR_TAKE(best)
        RR_TAKE(g_base) RR_TAKE(g_mask) RR_TAKE(t.base) RR_TAKE(t.hits) RR_TAKE(t.all)
        RR_TAKE(u_hits) RR_TAKE(sp)
#undef RR_TAKE
        const uint32_t qray = __shfl_sync(0xFFFFFFFFu, ray, from), qseg = __shfl_sync(0xFFFFFFFFu, seg, from);
        const LaneExtra<LEAN, BLOCK> owner{s_lane, (threadIdx.x & ~31u) + from, x.dir, x.second};
        RegisterExtra qx{owner.d(), owner.hit(), owner.u()};
        if (!LEAN) {
            qx.dir = make_float3(__shfl_sync(0xFFFFFFFFu, x.dir.x, from), __shfl_sync(0xFFFFFFFFu, x.dir.y, from),
                                 __shfl_sync(0xFFFFFFFFu, x.dir.z, from));
            qx.second = make_uint2(__shfl_sync(0xFFFFFFFFu, x.second.x, from), __shfl_sync(0xFFFFFFFFu, x.second.y, from));
        }
        bool qlive = left != 0u;
        while (__any_sync(0xFFFFFFFFu, qlive)) {
            const bool more = quad_step<ANY, BLOCK>(q, qx, qlive, stack, cx.scene(qseg), a.err, tables);
            if (qlive && !more && (lane & 3u) == 0u) cx.store(q, qx, qray, qseg);
            qlive = more;
        }
    }
    cx.leave();
}

// Few rays: four lanes to a ray from the start.
template <bool ACCUM, bool ANY, bool MULTI, int BLOCK>
__global__ void __launch_bounds__(BLOCK, 768 / BLOCK) trace_quad_kernel(TraceArgs a) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ QuantFrame s_frame;
    __shared__ float s_invE;
    __shared__ uint2 s_stack[kSharedStack * BLOCK];
    SceneRef *s_sc = reinterpret_cast<SceneRef *>(s_dyn);
    const TraceContext<ACCUM, MULTI> cx{a, s_sc, reinterpret_cast<uint32_t *>(s_sc + (MULTI ? a.n_segs : 0)), &s_frame,
                                        &s_invE};
    if (a.fills_device) allow_dependent_launch();
    const VisitTables &tables = block_visit_tables();
    wait_for_prerequisite();
    cx.load();
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31u, quad = lane >> 2;
    uint2 *stack = s_stack + (threadIdx.x & ~31u);
    RayState r;
    RegisterExtra x;
    x.begin(make_float4(0.0f, 0.0f, 0.0f, 0.0f));
    uint32_t ray = 0, seg = 0;
    bool live = false, exhausted = false;
    while (true) {
        const uint32_t idle = __ballot_sync(0xFFFFFFFFu, !live);
        if (!exhausted && idle != 0u) {
            // idle quads take consecutive queue positions
            const uint32_t want = (uint32_t)__popc(idle) >> 2;
            uint32_t base = 0;
            if (lane == 0) base = atomicAdd(a.queue, want);
            base = __shfl_sync(0xFFFFFFFFu, base, 0);
            if (base + want >= a.n) exhausted = true;
            if (!live && cx.find_ray(base + ((uint32_t)__popc(idle & ((1u << (4u * quad)) - 1u)) >> 2), ray, seg)) {
                ray_begin(r, x, cx.scene(seg), load_once(a.o_tmin + ray), load_once(a.d_tmax + ray));
                live = true;
            }
        }
        if (exhausted && __ballot_sync(0xFFFFFFFFu, live) == 0u) break;
        const bool more = quad_step_early<ANY, BLOCK>(r, x, live, stack, cx.scene(seg), a.err, tables);
        if (live && !more && (lane & 3u) == 0u) cx.store(r, x, ray, seg);
        live = more;
    }
    cx.leave();
}

}  // namespace rr

using namespace rr;

namespace {

DevNode device_node(const RRNode8 &n) {
    DevNode d{};
    d.px = n.px;
    d.py = n.py;
    d.pz = n.pz;
    d.masks = n.imask | n.valid << 8;
    const uint32_t s[3] = {(uint32_t)n.ex << 23, (uint32_t)n.ey << 23, (uint32_t)n.ez << 23};
    std::memcpy(&d.sx, &s[0], 4);
    std::memcpy(&d.sy, &s[1], 4);
    std::memcpy(&d.sz, &s[2], 4);
    d.child_base = n.child_base;
    std::memcpy(d.qlo_x, n.qlo_x, 8);
    std::memcpy(d.qlo_y, n.qlo_y, 8);
    std::memcpy(d.qlo_z, n.qlo_z, 8);
    std::memcpy(d.qhi_x, n.qhi_x, 8);
    std::memcpy(d.qhi_y, n.qhi_y, 8);
    std::memcpy(d.qhi_z, n.qhi_z, 8);
    d.tri_base = n.tri_base;
    d.tribits = n.tribits;
    return d;
}

RRNode8 host_node(const DevNode &d) {
    RRNode8 n{};
    n.px = d.px;
    n.py = d.py;
    n.pz = d.pz;
    n.imask = (uint8_t)d.masks;
    n.valid = d.masks >> 8;
    uint32_t s[3];
    std::memcpy(&s[0], &d.sx, 4);
    std::memcpy(&s[1], &d.sy, 4);
    std::memcpy(&s[2], &d.sz, 4);
    n.ex = (uint8_t)(s[0] >> 23);
    n.ey = (uint8_t)(s[1] >> 23);
    n.ez = (uint8_t)(s[2] >> 23);
    n.child_base = d.child_base;
    std::memcpy(n.qlo_x, d.qlo_x, 8);
    std::memcpy(n.qlo_y, d.qlo_y, 8);
    std::memcpy(n.qlo_z, d.qlo_z, 8);
    std::memcpy(n.qhi_x, d.qhi_x, 8);
    std::memcpy(n.qhi_y, d.qhi_y, 8);
    std::memcpy(n.qhi_z, d.qhi_z, 8);
    n.tri_base = d.tri_base;
    n.tribits = d.tribits;
    return n;
}

DevTri device_tri(const RRTri &t, const float4 *planes) {
    DevTri d;
    const float w[16] = {t.v0_id.x, t.v0_id.y, t.v0_id.z, t.e1.x,      t.e1.y,      t.e1.z,      t.e2.x,      t.e2.y,
                         t.e2.z,    t.v0_id.w, planes[0].x, planes[0].y, planes[0].z, planes[0].w, planes[1].x, planes[1].y};
    std::memcpy(&d, w, sizeof(d));
    return d;
}

void host_tri(const DevTri &d, const float *padding, RRTri *t, float4 *planes) {
    float id;
    std::memcpy(&id, &d.id, 4);
    t->v0_id = make_float4(d.v0[0], d.v0[1], d.v0[2], id);
    t->e1 = make_float4(d.e1[0], d.e1[1], d.e1[2], padding[0]);
    t->e2 = make_float4(d.e2[0], d.e2[1], d.e2[2], padding[1]);
    planes[0] = make_float4(d.nhi[0], d.nhi[1], d.nhi[2], d.nlo[0]);
    planes[1] = make_float4(d.nlo[1], d.nlo[2], padding[2], padding[3]);
}

// Whether a triangle's unused words hold anything but zero bits.
bool has_padding(const RRTri &t, const float4 &p1) {
    const float w[4] = {t.e1.w, t.e2.w, p1.z, p1.w}, zero[4] = {};
    return std::memcmp(w, zero, sizeof(w)) != 0;
}

// Uploads a host BVH into a new handle (synchronous).
rr_status upload_bvh(const HostBVH &h, uint32_t n_tris, double seconds, const char *what, rr_bvh **out) {
    rr_bvh *b = new rr_bvh();
    cudaGetDevice(&b->device);
    b->nodes = nullptr;
    b->tris = nullptr;
    b->n_nodes = (uint32_t)h.nodes.size();
    b->n_tris = n_tris;
    b->root_is_leaf = 0;
    b->root_leaf_ref = 0;
    cudaError_t e = cudaSuccess;
    if (b->n_nodes) {
        std::vector<DevNode> nodes(h.nodes.size());
        for (size_t i = 0; i < nodes.size(); ++i) nodes[i] = device_node(h.nodes[i]);
        std::vector<DevTri> tris(h.tris.size());
        for (size_t i = 0; i < tris.size(); ++i) tris[i] = device_tri(h.tris[i], &h.planes[2 * i]);
        bool padded = false;
        for (size_t i = 0; i < tris.size() && !padded; ++i) padded = has_padding(h.tris[i], h.planes[2 * i + 1]);
        if (padded)
            for (size_t i = 0; i < tris.size(); ++i)
                for (float x : {h.tris[i].e1.w, h.tris[i].e2.w, h.planes[2 * i + 1].z, h.planes[2 * i + 1].w})
                    b->padding.push_back(x);
        e = lib_malloc(reinterpret_cast<void **>(&b->nodes), sizeof(DevNode) * nodes.size());
        if (e == cudaSuccess) e = lib_malloc(reinterpret_cast<void **>(&b->tris), sizeof(DevTri) * tris.size());
        if (e == cudaSuccess)
            e = cudaMemcpy(b->nodes, nodes.data(), sizeof(DevNode) * nodes.size(), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(b->tris, tris.data(), sizeof(DevTri) * tris.size(), cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) {
        cudaFree(b->nodes);
        cudaFree(b->tris);
        delete b;
        cudaGetLastError();
        return fail(e == cudaErrorMemoryAllocation ? RR_ERR_OOM : RR_ERR_CUDA, std::string(what) + ": upload failed");
    }
    rr_bvh_info &i = b->info;
    i.n_tris = n_tris;
    i.n_nodes = b->n_nodes;
    i.n_leaves = h.n_leaves;
    i.depth = h.depth;
    i.node_bytes = sizeof(RRNode8) * (uint64_t)h.nodes.size();
    i.tri_bytes = sizeof(RRTri) * (uint64_t)h.tris.size() + sizeof(float4) * (uint64_t)h.planes.size();
    for (int c = 0; c < 3; ++c) {
        i.aabb_lo[c] = h.lo[c];
        i.aabb_hi[c] = h.hi[c];
    }
    i.build_seconds = seconds;
    *out = b;
    return RR_OK;
}

}  // namespace

extern "C" rr_status rr_build_bvh(const float *tris_host, uint32_t n_tris, rr_bvh **out) {
    if (!out) return fail(RR_ERR_INVALID_ARG, "rr_build_bvh: out is NULL");
    *out = nullptr;
    if (n_tris > 0 && !tris_host) return fail(RR_ERR_INVALID_ARG, "rr_build_bvh: tris is NULL");
    if (n_tris >= (1u << 28)) return fail(RR_ERR_UNSUPPORTED, "rr_build_bvh: at most 2^28 - 1 triangles");
    rr_status st;
    if (!device_state(&st)) return st;
    const auto t0 = std::chrono::steady_clock::now();
    HostBVH h;
    std::string err;
    st = build_wide_bvh(tris_host, n_tris, &h, &err);
    if (st != RR_OK) return fail(st, err);
    if (h.stack_need > kTraceStack)
        return fail(RR_ERR_UNSUPPORTED, "rr_build_bvh: tree needs a deeper traversal stack than the kernel has");
    return upload_bvh(h, n_tris, std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count(),
                      "rr_build_bvh", out);
}

extern "C" rr_status rr_bvh_serialize(const rr_bvh *b, void *buf, size_t *bytes) {
    if (!b || !bytes) return fail(RR_ERR_INVALID_ARG, "rr_bvh_serialize: NULL argument");
    const size_t need = serialized_bvh_bytes(b->n_nodes, b->n_tris);
    if (!buf) {
        *bytes = need;
        return RR_OK;
    }
    if (*bytes < need) {
        *bytes = need;
        return fail(RR_ERR_INVALID_ARG, "rr_bvh_serialize: buffer too small");
    }
    HostBVH h;
    h.nodes.resize(b->n_nodes);
    h.tris.resize(b->n_nodes ? b->n_tris : 0);
    h.planes.resize(2 * h.tris.size());
    cudaError_t e = cudaSuccess;
    if (b->n_nodes) {
        std::vector<DevNode> nodes(h.nodes.size());
        std::vector<DevTri> tris(h.tris.size());
        e = cudaMemcpy(nodes.data(), b->nodes, sizeof(DevNode) * nodes.size(), cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = cudaMemcpy(tris.data(), b->tris, sizeof(DevTri) * tris.size(), cudaMemcpyDeviceToHost);
        const float none[4] = {};
        for (size_t i = 0; i < nodes.size(); ++i) h.nodes[i] = host_node(nodes[i]);
        for (size_t i = 0; i < tris.size(); ++i)
            host_tri(tris[i], b->padding.empty() ? none : &b->padding[4 * i], &h.tris[i], &h.planes[2 * i]);
    }
    if (e != cudaSuccess) return fail_cuda(e, "rr_bvh_serialize: download");
    for (int c = 0; c < 3; ++c) {
        h.lo[c] = b->info.aabb_lo[c];
        h.hi[c] = b->info.aabb_hi[c];
    }
    h.depth = b->info.depth;
    h.n_leaves = b->info.n_leaves;
    serialize_bvh(h, buf);
    *bytes = need;
    return RR_OK;
}

extern "C" rr_status rr_bvh_deserialize(const void *buf, size_t bytes, rr_bvh **out) {
    if (!out) return fail(RR_ERR_INVALID_ARG, "rr_bvh_deserialize: out is NULL");
    *out = nullptr;
    rr_status st;
    if (!device_state(&st)) return st;
    HostBVH h;
    std::string err;
    st = deserialize_bvh(buf, bytes, &h, &err);
    if (st != RR_OK) return fail(st, err);
    return upload_bvh(h, (uint32_t)h.tris.size(), 0.0, "rr_bvh_deserialize", out);
}

extern "C" rr_status rr_bvh_destroy(rr_bvh *b) {
    if (!b) return RR_OK;
    cudaFree(b->nodes);
    cudaFree(b->tris);
    delete b;
    return RR_OK;
}

extern "C" rr_status rr_bvh_get_info(const rr_bvh *b, rr_bvh_info *info) {
    if (!b || !info) return fail(RR_ERR_INVALID_ARG, "rr_bvh_get_info: NULL argument");
    *info = b->info;
    return RR_OK;
}

extern "C" rr_status rr_bvh_aabb(const rr_bvh *b, float lo[3], float hi[3]) {
    if (!b || !lo || !hi) return fail(RR_ERR_INVALID_ARG, "rr_bvh_aabb: NULL argument");
    for (int c = 0; c < 3; ++c) {
        lo[c] = b->info.aabb_lo[c];
        hi[c] = b->info.aabb_hi[c];
    }
    return RR_OK;
}

namespace {

// Launches of at most this many rays put four lanes to a ray (two lanes are
// better than neither one nor four at any size).  Random order, one against four
// lanes, us; tiny scene: 4,097 rays 48 / 38, 8,192 49 / 40, 16,384 49 / 46, 25,000
// 53 / 56 (camera rays 16,384 36 / 37); 1,168,576 triangles: 16,384 85 / 74, 38,912
// 100 / 101.
constexpr uint32_t kQuadRays = 16384;

template <bool QUAD, bool ACC, bool ANY, bool MULTI, int BLOCK>
void *trace_entry() {
    return QUAD ? (void *)trace_quad_kernel<ACC, ANY, MULTI, BLOCK> : (void *)trace_kernel<ACC, ANY, MULTI, BLOCK>;
}

// Blocks of a trace kernel that an SM holds, and that shared-memory size: one
// word, so that callers on several threads see both of the same query.
template <bool QUAD, bool ACC, bool ANY, bool MULTI, int BLOCK>
cudaError_t trace_blocks_per_sm(size_t smem, uint32_t *blocks) {
    static std::atomic<uint64_t> known{0};  // smem << 16 | blocks
    const uint64_t k = known.load(std::memory_order_relaxed);
    if ((k & 0xFFFFu) != 0 && k >> 16 == smem) {  // the batch kernels' shared memory varies with the segments
        *blocks = (uint32_t)(k & 0xFFFFu);
        return cudaSuccess;
    }
    void *entry = trace_entry<QUAD, ACC, ANY, MULTI, BLOCK>();
    // Static and dynamic shared memory together may pass the default 48 KB: the
    // limit is raised before the query, which finds no room for a block beyond it
    // (one block per SM instead of two: 2M rays in 200 segments of a batch with
    // 512-thread blocks 1161 us instead of 740).
    if (MULTI) {
        const cudaError_t e = cudaFuncSetAttribute(entry, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)multi_smem(kMaxBatchSegments));
        if (e != cudaSuccess) return e;
    }
    int v = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, entry, BLOCK, smem);
    if (e != cudaSuccess) return e;
    *blocks = v < 1 ? 1u : (uint32_t)v;
    if (v >= 1) known.store((uint64_t)smem << 16 | (uint64_t)v, std::memory_order_relaxed);
    return cudaSuccess;
}

// An error stays the thread's last CUDA error, which the caller's check reports.
//
// Only a grid that fills the device lets the next kernel start early.  Beside a
// smaller one the next trace's blocks go where there is room, up to eight to an
// SM, instead of evenly, and stay there: traces of the tiny scene in a row,
// random order, 58,368 rays 86 us a launch instead of 59 (77,824, four blocks to
// an SM and room for four more, 64), 1,168,576 triangles any hit 49.5 instead of 36.
template <bool QUAD, bool ACC, bool ANY, bool MULTI, int BLOCK>
void trace_enqueue_form(TraceArgs a, int sm_count, cudaStream_t s) {
    const size_t smem = MULTI ? multi_smem(a.n_segs) : 0;
    const uint32_t per_block = QUAD ? BLOCK / 4 : BLOCK;  // rays a block holds at a time
    uint32_t bps = 0;
    if (trace_blocks_per_sm<QUAD, ACC, ANY, MULTI, BLOCK>(smem, &bps) != cudaSuccess) return;
    const uint32_t grid = std::max(1u, std::min((uint32_t)sm_count * bps, (a.n + per_block - 1u) / per_block));
    a.fills_device = grid == (uint32_t)sm_count * bps;
    launch_dependent(QUAD ? trace_quad_kernel<ACC, ANY, MULTI, BLOCK> : trace_kernel<ACC, ANY, MULTI, BLOCK>, grid, BLOCK,
                     smem, s, a);
}

template <bool ACC, bool ANY, bool MULTI, int BLOCK>
void trace_enqueue(const TraceArgs &a, int sm_count, cudaStream_t s) {
    if (a.n <= kQuadRays)
        trace_enqueue_form<true, ACC, ANY, MULTI, BLOCK>(a, sm_count, s);
    else
        trace_enqueue_form<false, ACC, ANY, MULTI, BLOCK>(a, sm_count, s);
}

rr_status launch_trace(const rr_bvh *b, const float *o_tmin, const float *d_tmax, const uint32_t *order, uint32_t n,
                       float *hits_out, uint32_t flags, rr_length_table *table, void *stream, const char *what) {
    if (!b) return fail(RR_ERR_INVALID_ARG, std::string(what) + ": NULL bvh");
    if (flags & ~(uint32_t)RR_TRACE_ANY_HIT) return fail(RR_ERR_INVALID_ARG, std::string(what) + ": unknown flags");
    const bool any = (flags & RR_TRACE_ANY_HIT) != 0;
    if (any && table)
        return fail(RR_ERR_INVALID_ARG, std::string(what) + ": any-hit distances are not ray lengths for the table");
    if (n == 0) return RR_OK;
    if (!o_tmin || !d_tmax || !hits_out) return fail(RR_ERR_INVALID_ARG, std::string(what) + ": NULL buffer");
    if (!aligned16(o_tmin) || !aligned16(d_tmax) || !aligned16(hits_out) || !aligned(order, 4))
        return fail(RR_ERR_INVALID_ARG, std::string(what) + ": misaligned buffer");
    if (overlaps(hits_out, 16ull * n, o_tmin, 16ull * n) || overlaps(hits_out, 16ull * n, d_tmax, 16ull * n) ||
        (order && overlaps(hits_out, 16ull * n, order, 4ull * n)))
        return fail(RR_ERR_INVALID_ARG, std::string(what) + ": hits overlap an input");
    rr_status st;
    DeviceState *ds = device_state(&st);
    if (!ds) return st;
    cudaStream_t s = as_stream(stream);
    TraceArgs a{};
    a.scene.nodes = b->nodes;
    a.scene.tris = b->tris;
    a.scene.n_nodes = b->n_nodes;
    a.scene.n_tris = b->n_tris;
    a.o_tmin = reinterpret_cast<const float4 *>(o_tmin);
    a.d_tmax = reinterpret_cast<const float4 *>(d_tmax);
    a.hits = reinterpret_cast<float4 *>(hits_out);
    a.order = order;
    a.n = n;
    a.err = error_word(ds, s);
    a.table = table ? table->cells : nullptr;
    for (int c = 0; c < 3; ++c) {
        a.tlo[c] = table ? table->box.lo[c] : 0.0f;
        a.thi[c] = table ? table->box.hi[c] : 0.0f;
    }
    // The length-table update: a separate pass over the traced rays when the
    // hits land in device memory (it runs at full lane use, with lanes that
    // share a cell combined before the atomics, and reads rays and hits from
    // L2), fused into the trace when they go straight to host memory.
    cudaPointerAttributes pa{};
    bool hits_on_device = false;
    if (table) {
        if (cudaPointerGetAttributes(&pa, hits_out) == cudaSuccess)
            hits_on_device = pa.type == cudaMemoryTypeDevice;
        else
            cudaGetLastError();
    }
    const bool fuse = table && !hits_on_device;
    const rr_status st2 = with_trace_queue(ds, s, [&](uint32_t *queue) {
        a.queue = queue;
        if (fuse)
            trace_enqueue<true, false, false, kTraceBlock>(a, ds->sm_count, s);
        else if (any)
            trace_enqueue<false, true, false, kTraceBlock>(a, ds->sm_count, s);
        else
            trace_enqueue<false, false, false, kTraceBlock>(a, ds->sm_count, s);
        note_launches(1);
        return check_launch(what);
    });
    if (st2 != RR_OK || !table || fuse) return st2;
    return rr_length_table_accumulate(table, o_tmin, d_tmax, hits_out, n, stream);
}

}  // namespace

namespace rr {

rr_status launch_trace_batch(const BatchScene *segs, const uint32_t *seg_offsets, uint32_t n_segs, const float *o_tmin,
                             const float *d_tmax, const uint32_t *order, uint32_t n, float *hits_out,
                             bool accumulate, uint32_t block, uint32_t *queue, uint32_t *err, cudaStream_t s) {
    rr_status st;
    DeviceState *ds = device_state(&st);
    if (!ds) return st;
    TraceArgs a{};
    a.o_tmin = reinterpret_cast<const float4 *>(o_tmin);
    a.d_tmax = reinterpret_cast<const float4 *>(d_tmax);
    a.hits = reinterpret_cast<float4 *>(hits_out);
    a.order = order;
    a.n = n;
    a.queue = queue;
    a.err = err;
    a.segs = segs;
    a.seg_offsets = seg_offsets;
    a.n_segs = n_segs;
    const int sms = ds->sm_count;
    if (accumulate) {
        if (block == 128) trace_enqueue<true, false, true, 128>(a, sms, s);
        else if (block == 512) trace_enqueue<true, false, true, 512>(a, sms, s);
        else trace_enqueue<true, false, true, 256>(a, sms, s);
    } else {
        if (block == 128) trace_enqueue<false, false, true, 128>(a, sms, s);
        else if (block == 512) trace_enqueue<false, false, true, 512>(a, sms, s);
        else trace_enqueue<false, false, true, 256>(a, sms, s);
    }
    note_launches(1);
    return check_launch("rr_batch trace");
}

}  // namespace rr

extern "C" rr_status rr_trace(const rr_bvh *b, const float *o_tmin, const float *d_tmax, uint32_t n, float *hits_out,
                              void *stream) {
    return launch_trace(b, o_tmin, d_tmax, nullptr, n, hits_out, 0u, nullptr, stream, "rr_trace");
}

extern "C" rr_status rr_trace_accumulate(const rr_bvh *b, const float *o_tmin, const float *d_tmax, uint32_t n,
                                         float *hits_out, rr_length_table *table, void *stream) {
    if (!table) return fail(RR_ERR_INVALID_ARG, "rr_trace_accumulate: NULL table");
    return launch_trace(b, o_tmin, d_tmax, nullptr, n, hits_out, 0u, table, stream, "rr_trace_accumulate");
}

extern "C" rr_status rr_trace_ex(const rr_bvh *b, const float *o_tmin, const float *d_tmax, const uint32_t *order,
                                 uint32_t n, float *hits_out, uint32_t flags, rr_length_table *table, void *stream) {
    return launch_trace(b, o_tmin, d_tmax, order, n, hits_out, flags, table, stream, "rr_trace_ex");
}
