// Narrow and broad phase of the edge-face detection (Sec. 3) and the
// penetration stencils (Sec. 4, Fig. 3).
//
// The broad phase (k_broad) walks the BVH of the oriented mesh's faces with
// every edge's box, testing both children of a node with one 64-byte node
// load, and lists the leaves met; the narrow phase (k_narrow) decides each by
// the exact segment-triangle test.  The edges are taken in the Morton order
// of their midpoints (a cached permutation), so that a warp walks one region
// of the tree.
// Hits are appended (one atomic per hit) as 64-bit keys
// (dir | edge | face), which a radix sort turns into the lexicographic
// (dir, v0, v1, face) order because the edges are sorted by (v0, v1).
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"
#include "predicates.cuh"
#include "sortdev.cuh"

namespace hfcr {

namespace {

constexpr int STACK = 64;

__device__ __forceinline__ int chk(int i, int n, uint32_t *st) {
    if ((unsigned)i < (unsigned)n) return i;
    atomicOr(st, ST_BAD_INDEX);
    return 0;
}

__device__ __forceinline__ bool overlap(const float *lo, const float *hi, float l0, float l1,
                                        float l2, float h0, float h1, float h2) {
    return lo[0] <= h0 && l0 <= hi[0] && lo[1] <= h1 && l1 <= hi[1] && lo[2] <= h2 && l2 <= hi[2];
}

__device__ __forceinline__ float lo_f(float v) { return v; }
__device__ __forceinline__ float hi_f(float v) { return v; }
__device__ __forceinline__ float lo_f(double v) { return __double2float_rd(v); }
__device__ __forceinline__ float hi_f(double v) { return __double2float_ru(v); }

template <typename T>
struct Leaf;
template <>
struct Leaf<float> {
    float a[3], b[3], c[3];
    int face;
    __device__ __forceinline__ void load(const void *base, int j) {
        const float4 *L = (const float4 *)base + 3 * j;
        float4 l0 = __ldg(L), l1 = __ldg(L + 1), l2 = __ldg(L + 2);
        a[0] = l0.x; a[1] = l0.y; a[2] = l0.z; b[0] = l0.w;
        b[1] = l1.x; b[2] = l1.y; c[0] = l1.z; c[1] = l1.w;
        c[2] = l2.x; face = __float_as_int(l2.y);
    }
};
template <>
struct Leaf<double> {
    double a[3], b[3], c[3];
    int face;
    __device__ __forceinline__ void load(const void *base, int j) {
        const double2 *L = (const double2 *)base + 5 * j;
        double2 l0 = __ldg(L), l1 = __ldg(L + 1), l2 = __ldg(L + 2), l3 = __ldg(L + 3),
                l4 = __ldg(L + 4);
        a[0] = l0.x; a[1] = l0.y; a[2] = l1.x; b[0] = l1.y;
        b[1] = l2.x; b[2] = l2.y; c[0] = l3.x; c[1] = l3.y;
        c[2] = l4.x; face = (int)__double_as_longlong(l4.y);
    }
};

template <typename T, bool F32F>
__device__ __forceinline__ bool leaf_test_body(const T *p, const T *q, const Leaf<T> &L, DevStats *st) {
    int side;
    if constexpr (F32F && sizeof(T) == 4) {
        f3 P = {(float)p[0], (float)p[1], (float)p[2]}, Q = {(float)q[0], (float)q[1], (float)q[2]};
        f3 A = {(float)L.a[0], (float)L.a[1], (float)L.a[2]};
        f3 B = {(float)L.b[0], (float)L.b[1], (float)L.b[2]};
        f3 C = {(float)L.c[0], (float)L.c[1], (float)L.c[2]};
        return segtri_f32(P, Q, A, B, C, side, st);
    } else {
        return segtri_f64<T>(p, q, L.a, L.b, L.c, side, st);
    }
}

// ---------------------------------------------------------------------------
// Broad phase: every warp keeps the pending visits of its edges (the edge's
// box, its index and a node) on one stack in shared memory and takes the
// newest 32 of them per step, one per lane, so an edge whose box overlaps
// thousands of faces is walked by the whole warp instead of by one lane while
// 31 wait.  While fewer than 32 visits are pending, the warp takes the next
// edges of the traversal order (its first ones are fixed, the others come
// from a device counter).  The leaves met, (edge, leaf), are appended to a
// list for the narrow phase (k_narrow), 32 at a time.
// Bound by the latency of dependent node loads and by how evenly the long
// walks spread: one thread per edge with the exact test inline needed 125
// registers (a quarter of the warps) and left a warp waiting for its longest
// walk.  Without the test this kernel needs 38 registers, and its lanes stay
// 95% busy.  Both phases against that form: a direction of 1,024 pairs of
// spheres of 80 to 20,480 faces 1.61 -> 0.56 ms, of two 262,144-face tori
// 50 -> 43 us, the 512 x 512 cloth over 327,680 faces 66 -> 50 us, the
// 200 x 200 cloth over 65,536 faces 64 -> 37 us, two 1,280-face float64
// spheres 131 -> 24 us.
// ---------------------------------------------------------------------------
constexpr int POOL_WARPS = 4;    // warps per CTA
constexpr int POOL_CAP = 128;    // pending visits in shared memory per warp
constexpr int POOL_SPILL = 128;  // blocks of 16 visits moved out to local memory at most
static_assert((POOL_CAP & (POOL_CAP - 1)) == 0 && POOL_CAP >= 64 + 16,
              "a step pushes up to 64 visits and moves out blocks of 16");

struct PoolSmem {
    float4 a[POOL_CAP];          // lo.xyz, hi.x
    float4 b[POOL_CAP];          // hi.yz, edge, node
    int2 leaf[32 + 64];          // fewer than 32 before a step, at most 64 more after it
};

// where the narrow phase puts its hits
struct HitList {
    unsigned long long *out;
    int *count;
    unsigned long long dirbit;
    int cap, face_bits;
    DevStats *st;
};
// the list between the two phases: n words of (edge, leaf), those beyond cap
// not stored
struct LeafList {
    int2 *items;
    int *n;
    int cap;
};

template <typename T>
__device__ __forceinline__ void edge_box(const T *p, const T *q, float *lo, float *hi) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lo[k] = lo_f(p[k] < q[k] ? p[k] : q[k]);
        hi[k] = hi_f(p[k] < q[k] ? q[k] : p[k]);
    }
}

// endpoints of an edge (out-of-range ids read vertex 0 and raise ST_BAD_INDEX)
template <typename T>
__device__ __forceinline__ void ld_edge(const int2 ev, const T *ex, const T *ey, const T *ez, int nv, T *p, T *q,
                                        uint32_t *status) {
    const int v0 = chk(ev.x, nv, status), v1 = chk(ev.y, nv, status);
    p[0] = ex[v0]; p[1] = ey[v0]; p[2] = ez[v0];
    q[0] = ex[v1]; q[1] = ey[v1]; q[2] = ez[v1];
}

// a node's 64 bytes by two 32-byte loads
__device__ __forceinline__ void ld_node(const float4 *nodes, int i, float *f) {
    const double4_32a *nd = (const double4_32a *)(nodes + 4 * (size_t)i);
    const double4_32a u = nd[0], v = nd[1];
    const double w[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        f[2 * k] = __int_as_float(__double2loint(w[k]));
        f[2 * k + 1] = __int_as_float(__double2hiint(w[k]));
    }
}

// what a walk is over: the edges of one direction and the trees they cross
template <typename T>
struct WalkArgs {
    const int2 *edges;
    const int *order;
    int ne, chunk;
    const T *ex, *ey, *ez;
    int nv;
    const float4 *nodes;
    int nfaces;
    const int *segs;
    int nseg, ecol, fcol;
    int *queue;  // edges taken beyond every warp's first
    uint32_t *status;
};

// One warp's share of the walk (CTAs of POOL_WARPS warps).  sink(leaves, n): n <=
// 32 leaves met, 32 of them but for the last of a batch; false ends the walk.
template <typename T, class Sink>
__device__ __forceinline__ void pool_walk(PoolSmem &sm, const WalkArgs<T> &g, Sink sink) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    int hint = 0;               // segment of this lane's last edge
    // pending visits: `n` of them in the ring ending at `top` (exclusive), and
    // `spilled` blocks of 16 older ones in local memory (lanes 0 to 15); nl
    // leaves wait (all the same in every lane)
    int top = 0, n = 0, nl = 0, spilled = 0;
    int2 spill[POOL_SPILL];
    int base = (blockIdx.x * POOL_WARPS + (threadIdx.x >> 5)) * g.chunk;  // the next edges
    // steps since the last edges were taken: guards against a corrupted tree
    // (an edge visits each of the 2 nfaces - 1 nodes at most once)
    unsigned steps = 0;
    const unsigned most = (unsigned)min(64ll * g.nfaces + 256, 0xffffffffll);
    while (true) {
        if (++steps > most) {
            if (lane == 0) atomicOr(g.status, ST_BAD_INDEX);
            break;
        }
        const bool fresh = n < 32 && spilled == 0 && base < g.ne;
        if (nl >= 32 || (nl > 0 && n == 0 && spilled == 0 && !fresh)) {
            const int take = min(nl, 32);
            nl -= take;
            if (!sink(sm.leaf + nl, take)) break;
            __syncwarp();
            continue;
        }
        bool on = false;
        float lo[3] = {0.f, 0.f, 0.f}, hi[3] = {0.f, 0.f, 0.f};
        int e = 0, node = 0;
        if (fresh) {
            const int i = base + lane;
            int t0 = 0, nleaf = 0;
            if (lane < g.chunk && i < g.ne) {
                e = g.order ? g.order[i] : i;
                const int2 ev = g.edges[e];
                if (g.nseg > 1 && !(g.segs[4 * hint + g.ecol] <= ev.x && ev.x < g.segs[4 * (hint + 1) + g.ecol]))
                    hint = seg_of(g.segs, g.ecol, g.nseg, ev.x);
                seg_range(g.segs, g.fcol, hint, g.nfaces, t0, nleaf);
                T p[3], q[3];
                ld_edge(ev, g.ex, g.ey, g.ez, g.nv, p, q, g.status);
                edge_box(p, q, lo, hi);
            }
            steps = 0;
            if (lane == 0) base = gridDim.x * POOL_WARPS * g.chunk + atomicAdd(g.queue, g.chunk);
            base = __shfl_sync(full, base, 0);
            const bool one = nleaf == 1;  // a tree of one leaf: tested outright
            const unsigned m = __ballot_sync(full, one);
            if (one) sm.leaf[nl + __popc(m & below)] = make_int2(e, t0);
            nl += __popc(m);
            on = nleaf > 1;
            node = t0;
        } else if (n > 0) {
            const int take = min(n, 32);
            on = lane < take;
            if (on) {
                const int at = (top - take + lane) & (POOL_CAP - 1);
                const float4 u = sm.a[at], w = sm.b[at];
                lo[0] = u.x; lo[1] = u.y; lo[2] = u.z; hi[0] = u.w;
                hi[1] = w.x; hi[2] = w.y;
                e = __float_as_int(w.z);
                node = __float_as_int(w.w);
            }
            top -= take;
            n -= take;
            __syncwarp();
        } else if (spilled > 0) {
            // a block of older visits back
            --spilled;
            if (lane < 16) {
                const int2 s = spill[spilled];
                T p[3], q[3];
                ld_edge(g.edges[s.x], g.ex, g.ey, g.ez, g.nv, p, q, g.status);
                edge_box(p, q, lo, hi);
                e = s.x;
                node = s.y;
                on = true;
            }
        } else {
            break;
        }
        // the visit: the node's two boxes against the edge's
        int c0 = 0, c1 = 0;
        bool h0 = false, h1 = false;
        if (on) {
            float f[16];
            ld_node(g.nodes, node, f);
            c0 = __float_as_int(f[12]);
            c1 = __float_as_int(f[13]);
            h0 = overlap(lo, hi, f[0], f[1], f[2], f[3], f[4], f[5]);
            h1 = overlap(lo, hi, f[6], f[7], f[8], f[9], f[10], f[11]);
        }
        const unsigned l0 = __ballot_sync(full, h0 && c0 < 0), l1 = __ballot_sync(full, h1 && c1 < 0);
        if (l0 | l1) {
            if (h0 && c0 < 0) sm.leaf[nl + __popc(l0 & below)] = make_int2(e, ~c0);
            if (h1 && c1 < 0) sm.leaf[nl + __popc(l0) + __popc(l1 & below)] = make_int2(e, ~c1);
            nl += __popc(l0) + __popc(l1);
        }
        const unsigned i0 = __ballot_sync(full, h0 && c0 >= 0), i1 = __ballot_sync(full, h1 && c1 >= 0);
        const int add = __popc(i0) + __popc(i1);
        while (n + add > POOL_CAP) {  // the 16 oldest visits out of the ring
            if (lane < 16) {
                const float4 s = sm.b[(top - n + lane) & (POOL_CAP - 1)];
                if (spilled < POOL_SPILL) spill[spilled] = make_int2(__float_as_int(s.z), __float_as_int(s.w));
                else atomicOr(g.status, ST_BAD_INDEX);  // unreachable: depth < 64
            }
            spilled = min(spilled + 1, POOL_SPILL);
            n -= 16;
            __syncwarp();
        }
        const float4 u = make_float4(lo[0], lo[1], lo[2], hi[0]);
        if (h0 && c0 >= 0) {
            const int at = (top + __popc(i0 & below)) & (POOL_CAP - 1);
            sm.a[at] = u;
            sm.b[at] = make_float4(hi[1], hi[2], __int_as_float(e), __int_as_float(c0));
        }
        if (h1 && c1 >= 0) {
            const int at = (top + __popc(i0) + __popc(i1 & below)) & (POOL_CAP - 1);
            sm.a[at] = u;
            sm.b[at] = make_float4(hi[1], hi[2], __int_as_float(e), __int_as_float(c1));
        }
        top += add;
        n += add;
        __syncwarp();
    }
}

// Once the list is over its capacity the count stays there and the warps
// leave: k_narrow then walks on its own.
template <typename T>
__global__ void __launch_bounds__(32 * POOL_WARPS, 8) k_broad(WalkArgs<T> g, LeafList out) {
    HFCR_PDL_WAIT();
    // malformed input (reported by the host): its tree is not walked
    if (__any_sync(0xffffffffu, (*(volatile uint32_t *)g.status & ST_BAD_INDEX) != 0)) return;
    __shared__ PoolSmem smw[POOL_WARPS];
    pool_walk(smw[threadIdx.x >> 5], g, [&](const int2 *leaf, int take) {
        const int lane = threadIdx.x & 31;
        int at = 0;
        if (lane == 0) {
            at = *(volatile int *)out.n;
            if (at <= out.cap) at = atomicAdd(out.n, take);
        }
        at = __shfl_sync(0xffffffffu, at, 0);
        if (lane < take && at + lane < out.cap) out.items[at + lane] = leaf[lane];
        return at <= out.cap;
    });
}

// leaf lf against an edge, the hit appended
template <typename T, bool F32F>
__device__ __forceinline__ void narrow_test(const T *p, const T *q, int e, int lf, const void *leaf_tri,
                                            const HitList &o) {
    Leaf<T> L;
    L.load(leaf_tri, lf);
    if (leaf_test_body<T, F32F>(p, q, L, o.st)) {
        const int pos = atomicAdd(o.count, 1);
        if (pos < o.cap)
            o.out[pos] = o.dirbit | ((unsigned long long)e << o.face_bits) | (unsigned)L.face;
    }
}

// the same out of line
template <typename T, bool F32F>
__device__ __noinline__ void narrow_test_call(const int2 l, const WalkArgs<T> &g, const void *leaf_tri,
                                              const HitList &o) {
    T p[3], q[3];
    ld_edge(g.edges[l.x], g.ex, g.ey, g.ez, g.nv, p, q, g.status);
    narrow_test<T, F32F>(p, q, l.x, l.y, leaf_tri, o);
}

// Narrow phase: the exact test of every (edge, leaf) of the broad phase, one
// per thread, consecutive warps' work on different CTAs (few tests spread
// over many SMs: the float64 stages are slow on one).  When the list
// overflowed, it walks the edges itself as the broad phase does and tests
// the leaves 32 at a time as they are met.
template <typename T, bool F32F>
__global__ void __launch_bounds__(32 * POOL_WARPS) k_narrow(const __grid_constant__ WalkArgs<T> g,
                                                            const void *leaf_tri,
                                                            const __grid_constant__ HitList o, LeafList in) {
    HFCR_PDL_WAIT();
    if (*(volatile uint32_t *)g.status & ST_BAD_INDEX) return;
    const int n = *in.n, lane = threadIdx.x & 31;
    if (n <= in.cap) {
        const int first = ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + lane;
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&o.st->narrow_tests, (unsigned long long)n);
        for (int i = first; i < n; i += gridDim.x * 128) {
            const int2 l = in.items[i];
            T p[3], q[3];
            ld_edge(g.edges[l.x], g.ex, g.ey, g.ez, g.nv, p, q, g.status);
            narrow_test<T, F32F>(p, q, l.x, l.y, leaf_tri, o);
        }
        return;
    }
    __shared__ PoolSmem smw[POOL_WARPS];
    unsigned tests = 0;
    pool_walk(smw[threadIdx.x >> 5], g, [&](const int2 *leaf, int take) {
        if (lane < take) narrow_test_call<T, F32F>(leaf[lane], g, leaf_tri, o);
        tests += take;
        return true;
    });
    if (lane == 0 && tests) atomicAdd(&o.st->narrow_tests, (unsigned long long)tests);
}

__global__ void k_keys_to_pairs(const unsigned long long *keys, const int *d_n, int cap,
                                const int2 *edgesA, const int2 *edgesB, int edge_bits,
                                int face_bits, hfcr_pair *out) {
    HFCR_PDL_WAIT();
    int n = min(*d_n, cap);
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned long long k = keys[i];
    unsigned dir = (unsigned)(k >> (edge_bits + face_bits));
    unsigned e = (unsigned)((k >> face_bits) & ((1ull << edge_bits) - 1));
    unsigned f = (unsigned)(k & ((1ull << face_bits) - 1));
    int2 ev = dir ? edgesB[e] : edgesA[e];
    out[i] = hfcr_pair{dir, (unsigned)ev.x, (unsigned)ev.y, f};
}

template <typename T>
__device__ __forceinline__ void ld3(const hfcr_mesh &m, int i, T *o) {
    o[0] = ((const T *)m.x)[i];
    o[1] = ((const T *)m.y)[i];
    o[2] = ((const T *)m.z)[i];
}

// x0 = the endpoint of the pair's edge on the back side of its face
// stencil key of the pair (dir, v0, v1, f): x0 = the endpoint of the edge on
// the back side of its face
template <typename T>
__device__ __forceinline__ unsigned long long stencil_key_of(const hfcr_mesh &A, const hfcr_mesh &B,
                                                             unsigned dir, unsigned pv0, unsigned pv1,
                                                             unsigned pf, int vert_bits, int face_bits,
                                                             int f32_filter, DevStats *st,
                                                             uint32_t *status) {
    const hfcr_mesh &E = dir ? B : A;
    const hfcr_mesh &F = dir ? A : B;
    int v0 = chk((int)pv0, E.n_verts, status), v1 = chk((int)pv1, E.n_verts, status);
    int f = chk((int)pf, F.n_tris, status);
    int ia = chk(F.tris[3 * f], F.n_verts, status), ib = chk(F.tris[3 * f + 1], F.n_verts, status),
        ic = chk(F.tris[3 * f + 2], F.n_verts, status);
    T a[3], b[3], c[3], p[3];
    ld3<T>(F, ia, a);
    ld3<T>(F, ib, b);
    ld3<T>(F, ic, c);
    ld3<T>(E, v0, p);
    int s = orient_full<T>(a, b, c, p, f32_filter, st);
    // a crossing pair has s != 0; a pair given by the caller with the first
    // endpoint on the plane keeps v1 (the crossing test would reject it)
    unsigned x0 = s < 0 ? (unsigned)v0 : (unsigned)v1;
    return ((unsigned long long)dir << (vert_bits + face_bits)) |
           ((unsigned long long)x0 << face_bits) | (unsigned long long)(unsigned)f;
}

template <typename T>
__global__ void k_stencil_keys(hfcr_mesh A, hfcr_mesh B, const hfcr_pair *pairs, const int *d_n,
                               int cap, int vert_bits, int face_bits, int f32_filter,
                               unsigned long long *keys, DevStats *st, uint32_t *status) {
    HFCR_PDL_WAIT();
    int n = min(*d_n, cap);
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    hfcr_pair pr = pairs[i];
    unsigned dir = pr.dir ? 1u : 0u;
    if (pr.dir > 1u) atomicOr(status, ST_BAD_INDEX);
    keys[i] = stencil_key_of<T>(A, B, dir, pr.v0, pr.v1, pr.face, vert_bits, face_bits, f32_filter,
                                st, status);
}

// The same from the traversal's pair keys (dir | edge | face) as appended:
// the pair count is clamped here (more than cap: ST_CAPACITY and no pair;
// the clamped count to *d_eff for the kernels that follow)
template <typename T>
__global__ void k_stencil_keys_from_pair_keys(hfcr_mesh A, hfcr_mesh B,
                                              const unsigned long long *pkeys, const int *d_n,
                                              int cap, const int2 *edgesA, const int2 *edgesB,
                                              int edge_bits, int pface_bits, int vert_bits,
                                              int face_bits, int f32_filter,
                                              unsigned long long *keys, int *d_eff, DevStats *st,
                                              uint32_t *status) {
    HFCR_PDL_WAIT();
    int n = *d_n;
    if (n > cap) n = 0;
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        if (*d_n > cap) atomicOr(status, ST_CAPACITY);
        *d_eff = n;
    }
    if (i >= n) return;
    const unsigned long long k = pkeys[i];
    const unsigned dir = (unsigned)(k >> (edge_bits + pface_bits));
    const int e = (int)((k >> pface_bits) & ((1ull << edge_bits) - 1));
    const unsigned f = (unsigned)(k & ((1ull << pface_bits) - 1));
    const int2 ev = dir ? edgesB[e] : edgesA[e];
    keys[i] = stencil_key_of<T>(A, B, dir, (unsigned)ev.x, (unsigned)ev.y, f, vert_bits, face_bits,
                                f32_filter, st, status);
}

// sorted keys -> the list of distinct ones, their number to *d_k: one
// single-pass scan (lookback), UNIQUE_KEYS keys per CTA, in the place of flags,
// their two-kernel scan and the write
constexpr int UNIQUE_KEYS = 1024;

__global__ void __launch_bounds__(TPB) k_stencil_unique(const unsigned long long *many,
                                                        const unsigned long long *few, const int *d_n, int cap,
                                                        int vert_bits, int face_bits, hfcr_stencil *out, int *d_k,
                                                        int *ticket, unsigned long long *state,
                                                        uint32_t *status) {
    HFCR_PDL_WAIT();
    const int n = min(*d_n, cap);
    const unsigned long long *keys = n <= RANK_MAX ? few : many;
    __shared__ int cta;
    __shared__ unsigned ws[TPB / 32], base;
    if ((int)blockIdx.x * UNIQUE_KEYS >= n) {  // nothing for it (the tickets below are the others')
        if (blockIdx.x == 0 && threadIdx.x == 0) *d_k = 0;
        return;
    }
    if (threadIdx.x == 0) cta = atomicAdd(ticket, 1);
    __syncthreads();
    constexpr int PER = UNIQUE_KEYS / TPB;
    const int i0 = cta * UNIQUE_KEYS + threadIdx.x * PER;
    unsigned long long k[PER + 1];
    k[0] = i0 > 0 && i0 <= n ? keys[i0 - 1] : ~0ull;  // no key has every bit set
#pragma unroll
    for (int q = 0; q < PER; ++q) k[q + 1] = i0 + q < n ? keys[i0 + q] : k[q];
    unsigned sum = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) sum += k[q + 1] != k[q];
    unsigned total;
    unsigned at = cta_scan(sum, ws, total);
    if (threadIdx.x < 32) {
        const unsigned b = lookback(state, cta, total, status);
        if (threadIdx.x == 0) {
            base = b;
            if ((cta + 1) * UNIQUE_KEYS >= n) *d_k = (int)(b + total);
        }
    }
    __syncthreads();
    at += base;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        if (k[q + 1] == k[q]) continue;
        const unsigned long long v = k[q + 1];
        hfcr_stencil s;
        s.dir = (unsigned)(v >> (vert_bits + face_bits));
        s.x0 = (unsigned)((v >> face_bits) & ((1ull << vert_bits) - 1));
        s.face = (unsigned)(v & ((1ull << face_bits) - 1));
        s.pad = 0;
        out[at++] = s;
    }
}

// effective count = count when it fits the capacity, else 0 with
// ST_CAPACITY raised (so nothing downstream runs on a truncated set)
__device__ __forceinline__ int first_edge_from(const int2 *E, int ne, int v) {
    int lo = 0, hi = ne;  // first edge whose first vertex is >= v
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (E[mid].x < v) lo = mid + 1; else hi = mid;
    }
    return lo;
}

__global__ void k_pair_products(const int2 *E, int ne, const int *segs, int nseg, int ecol, int fcol,
                                int nfaces, DevStats *st) {
    HFCR_PDL_WAIT();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long v = 0;
    if (i < nseg) {
        int e0 = first_edge_from(E, ne, segs[4 * i + ecol]);
        int e1 = first_edge_from(E, ne, segs[4 * (i + 1) + ecol]);
        int f0, nf;
        seg_range(segs, fcol, i, nfaces, f0, nf);
        v = (unsigned long long)max(e1 - e0, 0) * (unsigned long long)nf;
    }
    v = __reduce_add_sync(0xffffffffu, (unsigned)(v & 0xffffffffu)) +
        ((unsigned long long)__reduce_add_sync(0xffffffffu, (unsigned)(v >> 32)) << 32);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(&st->bf, v);
}

}  // namespace

void pair_products(const int *edges, int ne, const int *segs, int nseg, int ecol, int fcol,
                   int nfaces, DevStats *stats, cudaStream_t s) {
    if (ne <= 0 || nseg <= 0) return;
    { launch_pdl(k_pair_products, (nseg + 255) / 256, 256, 0, s, (const int2 *)edges, ne, segs,
                 nseg, ecol,
                                                        fcol, nfaces, stats); note_launch(); }
}

// resident CTAs of the broad phase on this device (cached)
template <typename T>
static int broad_ctas() {
    static int dev_cache[64];
    static bool done[64];
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return 152;
    if (!done[dev]) {
        int sms = 0, per = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_broad<T>, 32 * POOL_WARPS, 0);
        dev_cache[dev] = sms * (per > 0 ? per : 1);
        done[dev] = true;
    }
    return dev_cache[dev];
}

template <typename T, bool F32F>
static void launch_phases(const DetectArgs &a, cudaStream_t s, uint32_t *d_status) {
    const hfcr_mesh &m = *a.edge_mesh;
    const T *x = (const T *)m.x, *y = (const T *)m.y, *z = (const T *)m.z;
    const unsigned long long dirbit = (unsigned long long)a.dir << (a.edge_bits + a.face_bits);
    // the variant: 32, 16 or 8 edges taken at a time, on all, 3/4 or half of
    // the CTAs that fit; with few edges fewer at a time, so that every warp
    // has some (down to 4: a tree's levels are walked one after the other
    // however few edges a warp has)
    int grid = broad_ctas<T>() * (4 - a.variant / 3) / 4;
    if (grid < 1) grid = 1;
    const int most = 32 >> (a.variant % 3);
    int chunk = (a.n_edges + grid * POOL_WARPS - 1) / (grid * POOL_WARPS);
    chunk = chunk < 4 ? 4 : (chunk > most ? most : chunk);
    const int need = (a.n_edges + chunk * POOL_WARPS - 1) / (chunk * POOL_WARPS);
    if (grid > need) grid = need;
    const LeafList l = {a.leaves, a.queue + 1, a.leaf_cap};
    WalkArgs<T> g = {(const int2 *)a.edges, a.order, a.n_edges, chunk, x, y, z, m.n_verts, a.bvh->nodes,
                     a.bvh->n, a.segs, a.nseg, a.ecol, a.fcol, a.queue, d_status};
    { launch_pdl(k_broad<T>, grid, 32 * POOL_WARPS, 0, s, g, l); note_launch(); }
    const HitList o = {a.keys, a.d_count, dirbit, a.cap, a.face_bits, a.stats};
    int gn = (a.n_edges + 127) / 128;
    if (gn > 8 * 152) gn = 8 * 152;
    g.queue = a.queue + 2;
    { launch_pdl(k_narrow<T, F32F>, gn, 32 * POOL_WARPS, 0, s, g, (const void *)a.bvh->leaf_tri, o, l);
      note_launch(); }
}

void detect_launch(const DetectArgs &a, cudaStream_t s, uint32_t *d_status) {
    if (a.n_edges <= 0 || a.bvh->n <= 0) return;
    if (a.edge_mesh->dtype != HFCR_F32) launch_phases<double, false>(a, s, d_status);
    else if (a.f32_filter) launch_phases<float, true>(a, s, d_status);
    else launch_phases<float, false>(a, s, d_status);
}

void keys_to_pairs(const unsigned long long *keys, const int *d_n, int cap, const int *edgesA,
                   const int *edgesB, int edge_bits, int face_bits, hfcr_pair *out, cudaStream_t s) {
    if (cap <= 0) return;
    { launch_pdl(k_keys_to_pairs, (cap + 255) / 256, 256, 0, s, keys, d_n, cap,
                 (const int2 *)edgesA,
                                                      (const int2 *)edgesB, edge_bits, face_bits, out); note_launch(); }
}

void stencil_keys(const MeshPair &mp, const hfcr_pair *pairs, const int *d_n, int cap,
                  int vert_bits, int face_bits, int f32_filter, unsigned long long *keys,
                  DevStats *stats, uint32_t *d_status, cudaStream_t s) {
    if (cap <= 0) return;
    int nb = (cap + 255) / 256;
    if (mp.A.dtype == HFCR_F32)
        { launch_pdl(k_stencil_keys<float>, nb, 256, 0, s, mp.A, mp.B, pairs, d_n, cap, vert_bits,
                     face_bits,
                                                 f32_filter, keys, stats, d_status); note_launch(); }
    else
        { launch_pdl(k_stencil_keys<double>, nb, 256, 0, s, mp.A, mp.B, pairs, d_n, cap,
                     vert_bits, face_bits,
                                                  f32_filter, keys, stats, d_status); note_launch(); }
}

void stencil_keys_from_pair_keys(const MeshPair &mp, const unsigned long long *pkeys, const int *d_n,
                                 int cap, const int *edgesA, const int *edgesB, int edge_bits,
                                 int pface_bits, int vert_bits, int face_bits, int f32_filter,
                                 unsigned long long *keys, int *d_eff, DevStats *stats,
                                 uint32_t *d_status, cudaStream_t s) {
    if (cap <= 0) return;
    const int nb = (cap + 255) / 256;
    if (mp.A.dtype == HFCR_F32)
        launch_pdl(k_stencil_keys_from_pair_keys<float>, nb, 256, 0, s, mp.A, mp.B, pkeys, d_n, cap,
                   (const int2 *)edgesA, (const int2 *)edgesB, edge_bits, pface_bits, vert_bits,
                   face_bits, f32_filter, keys, d_eff, stats, d_status);
    else
        launch_pdl(k_stencil_keys_from_pair_keys<double>, nb, 256, 0, s, mp.A, mp.B, pkeys, d_n, cap,
                   (const int2 *)edgesA, (const int2 *)edgesB, edge_bits, pface_bits, vert_bits,
                   face_bits, f32_filter, keys, d_eff, stats, d_status);
    note_launch();
}

void stencil_unique(const unsigned long long *keys, const unsigned long long *few, const int *d_n, int cap,
                    int vert_bits, int face_bits, hfcr_stencil *out, int *d_k, int *words,
                    uint32_t *d_status, cudaStream_t s) {
    if (cap <= 0) return;
    { launch_pdl(k_stencil_unique, (cap + UNIQUE_KEYS - 1) / UNIQUE_KEYS, TPB, 0, s, keys, few, d_n, cap,
                 vert_bits, face_bits, out, d_k, words, (unsigned long long *)(words + 2), d_status);
      note_launch(); }
}

}  // namespace hfcr
