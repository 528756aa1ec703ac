// Topology (edges), input validation and the linear BVH over the faces of
// an oriented mesh.
//
// The paper only says that detection uses tight bounding volumes (Sec. 1);
// the hierarchy here is a binary radix tree over 30-bit Morton codes of the
// face centroids (Karras 2012), refitted bottom-up: block by block in shared
// memory, then the few nodes that span blocks.
// Boxes are float32 and conservative: for float32 coordinates min/max are
// exact, for float64 they are rounded outward, so box rejection never drops
// a true intersection.
#include <cuda_runtime.h>
#include <float.h>
#include <stdint.h>

#include "internal.h"
#include "sortdev.cuh"

namespace hfcr {

namespace {

// segment table sanity: rows non-decreasing, first row 0, last row equal to
// the mesh sizes (the concatenated A and B)
__global__ void k_check_segs(const int *segs, int nseg, int nva, int nta, int nvb, int ntb,
                             uint32_t *st) {
    HFCR_PDL_WAIT();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i > nseg) return;
    const int tot[4] = {nva, nta, nvb, ntb};
    for (int c = 0; c < 4; ++c) {
        int v = segs[4 * i + c];
        bool bad = (i == 0 && v != 0) || (i == nseg && v != tot[c]) ||
                   (i > 0 && v < segs[4 * (i - 1) + c]) || v < 0 || v > tot[c];
        if (bad) atomicOr(st, ST_BAD_INDEX);
    }
}

// index into [0, n): out-of-range ids read element 0 and raise ST_BAD_INDEX
__device__ __forceinline__ int chk(int i, int n, uint32_t *st) {
    if ((unsigned)i < (unsigned)n) return i;
    atomicOr(st, ST_BAD_INDEX);
    return 0;
}

template <typename T>
__global__ void k_validate(const T *x, const T *y, const T *z, int n, uint32_t *status) {
    HFCR_PDL_WAIT();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t bad = 0;
    if (i < n) {
        T c[3] = {x[i], y[i], z[i]};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            T v = c[k];
            if (!isfinite(v)) {
                bad |= ST_NONFINITE;
            } else {
                T a = fabs(v);
                if (a > (T)0x1p38) bad |= ST_RANGE;
                if (sizeof(T) == 8 && a != (T)0 && a < (T)0x1p-200) bad |= ST_RANGE;
            }
        }
    }
    bad = __reduce_or_sync(0xffffffffu, bad);
    if (bad && (threadIdx.x & 31) == 0) atomicOr(status, bad);
}

// both meshes of a pair in one launch: vertex i < nA of A, else i - nA of B
template <typename T>
__global__ void k_validate_pair(const T *ax, const T *ay, const T *az, int nA, const T *bx,
                                const T *by, const T *bz, int nB, uint32_t *status) {
    HFCR_PDL_WAIT();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t bad = 0;
    if (i < nA + nB) {
        const bool inA = i < nA;
        const int j = inA ? i : i - nA;
        T c[3] = {inA ? ax[j] : bx[j], inA ? ay[j] : by[j], inA ? az[j] : bz[j]};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            T v = c[k];
            if (!isfinite(v)) {
                bad |= ST_NONFINITE;
            } else {
                T a = fabs(v);
                if (a > (T)0x1p38) bad |= ST_RANGE;
                if (sizeof(T) == 8 && a != (T)0 && a < (T)0x1p-200) bad |= ST_RANGE;
            }
        }
    }
    bad = __reduce_or_sync(0xffffffffu, bad);
    if (bad && (threadIdx.x & 31) == 0) atomicOr(status, bad);
}

__global__ void k_edge_keys(const int *tris, int nt, int vb, unsigned long long *keys,
                            uint32_t *status, int nv) {
    HFCR_PDL_WAIT();
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    int v[3] = {tris[3 * t], tris[3 * t + 1], tris[3 * t + 2]};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int a = v[k], b = v[(k + 1) % 3];
        if ((unsigned)a >= (unsigned)nv || (unsigned)b >= (unsigned)nv) {
            atomicOr(status, ST_BAD_INDEX);
            a = b = 0;
        }
        unsigned long long lo = (unsigned)min(a, b), hi = (unsigned)max(a, b);
        keys[3 * t + k] = (lo << vb) | hi;
    }
}

__global__ void k_unique_flags(const unsigned long long *keys, int n, unsigned *flags) {
    HFCR_PDL_WAIT();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) flags[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1u : 0u;
}

__global__ void k_write_edges(const unsigned long long *keys, const unsigned *pos, int n, int vb,
                              int *edges) {
    HFCR_PDL_WAIT();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (i == 0 || keys[i] != keys[i - 1]) {
        unsigned long long k = keys[i];
        unsigned p = pos[i];
        edges[2 * p] = (int)(k >> vb);
        edges[2 * p + 1] = (int)(k & ((1ull << vb) - 1));
    }
}

// ---- the edges of a triangle list by buckets of the smaller vertex ----
//
// Four kernels instead of a radix sort of the 3 n_tris (v0, v1) keys: the
// half-edges are counted per v0 (each keeps the rank the counter gave it), the
// counts scanned, the v1 placed, and each vertex's v1 sorted and made unique.
// The few of an ordinary vertex (a manifold mesh has some twelve) by one
// thread in shared memory; with HUBS up to BUCKET_WARP by a warp (ranks), and
// the list of a hub (a fan, a pole) by the CTA through a bitmap.  Whatever the
// form does not take raises *slow: without HUBS a vertex of more than
// BUCKET_SHORT half-edges, with them a block of vertices that has more long
// lists than the sort would cost, or a vertex of more half-edges than a rank
// holds.  The caller then tries the next form, at last the sort
// (build_edges_sorted), which does not care.  Both scans are single-pass: a
// CTA publishes its sum and looks back over its predecessors' (tickets in
// starting order, so they are running).
// 522,242 triangles: 166 us of kernels by the sort (five passes of scattered
// 8-byte keys), 45 by buckets; whole calls 158 and 55 us, and 59 with HUBS,
// which costs nothing that shows up to BUCKET_HUBS_TRIS.
// With a pole of 200 half-edges, 10,000 triangles: 238 us by the sort, 40 with
// HUBS; of 1,024, 262,144 triangles: 112 by the sort, 82 by both tries.  A call
// that ends at the sort has paid about 20 us for the tries (a fan of 20,000
// triangles 106 us, 85 by the sort alone).
constexpr int BUCKET_SHORT = 32;         // sorted by one thread: 256 moves of some 30 cycles
constexpr int BUCKET_WARP = 128;         // by a warp: n^2 / 32 comparisons
constexpr int BUCKET_RANK = 65535;       // a hub's half-edges at most
constexpr int BUCKET_HUBS_TRIS = 100000; // triangles of a mesh whose first try has HUBS
constexpr int BUCKET_SM = 3968;          // v1 of one CTA's vertices kept in shared memory (six CTAs per SM)
constexpr int BUCKET_TPB = TPB;
constexpr int BUCKET_SCAN = 2048;        // counts per CTA of the scan
static_assert(BUCKET_SCAN / BUCKET_TPB * 32 == BUCKET_TPB, "a warp of the scan has the counts of one CTA of k_bucket_edges");

// Cycles, roughly, that a CTA of k_bucket_edges spends on a list of n half-
// edges beyond an ordinary one's, one of its eight warps (measured: 780 at 34,
// 3,700 at 120) or the whole CTA (5,500 at 1,000, more where the ids spread over
// further passes of the bitmap), and what the sort costs more
// than the buckets do, their own start and the read-back among it: 60 vertices
// of 34 half-edges in a block 61 us either way, one of 30,000 85.
__device__ __forceinline__ unsigned bucket_cost(unsigned n, unsigned passes) {
    return n <= (unsigned)BUCKET_WARP ? 600 + n * n / 5 : 15000 * passes - 12500 + 3 * n;
}
__device__ __forceinline__ unsigned bucket_cost_limit(unsigned n_tris) { return 100000 + n_tris / 8; }

template <bool HUBS>
struct BucketRank { typedef unsigned char T; };
template <>
struct BucketRank<true> { typedef uint16_t T; };

template <bool HUBS>
__global__ void __launch_bounds__(BUCKET_TPB) k_bucket_count(const int *tris, int nt, int nv, int *cnt,
                                                             typename BucketRank<HUBS>::T *rank, int *slow,
                                                             uint32_t *status) {
    HFCR_PDL_WAIT();
    const int t = blockIdx.x * BUCKET_TPB + threadIdx.x;
    const unsigned live = __ballot_sync(0xffffffffu, t < nt);
    if (t >= nt) return;
    const int v[3] = {tris[3 * t], tris[3 * t + 1], tris[3 * t + 2]};
    int u[3], r[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int a = v[k], b = v[(k + 1) % 3];
        if ((unsigned)a >= (unsigned)nv || (unsigned)b >= (unsigned)nv) {
            atomicOr(status, ST_BAD_INDEX);
            a = b = 0;
        }
        u[k] = min(a, b);
    }
    bool hubs = false;
    if constexpr (HUBS) {
        // around a hub a warp's triangles all have it: one addition for its two
        // half-edges of each
        const int hub = min(u[0], min(u[1], u[2])), first = __ffs(live) - 1;
        const int hub0 = __shfl_sync(live, hub, first);
        hubs = __all_sync(live, hub == hub0 && (u[0] == hub) + (u[1] == hub) + (u[2] == hub) == 2);
        if (hubs) {
            const int lane = threadIdx.x & 31;
            int base = 0;
            if (lane == first) base = atomicAdd(cnt + hub, 2 * __popc(live));
            base = __shfl_sync(live, base, first) + 2 * __popc(live & ((1u << lane) - 1u));
#pragma unroll
            for (int k = 0; k < 3; ++k) r[k] = u[k] == hub ? base++ : atomicAdd(cnt + u[k], 1);
        }
    }
    if (!hubs) {
#pragma unroll
        for (int k = 0; k < 3; ++k) r[k] = atomicAdd(cnt + u[k], 1);
    }
    constexpr int most = HUBS ? BUCKET_RANK : BUCKET_SHORT;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (r[k] >= most) *slow = 1;
        rank[3 * t + k] = (typename BucketRank<HUBS>::T)min(r[k], most);
    }
}

// cnt[0 .. n) -> exclusive offsets in place, the total to cnt[n]
template <bool HUBS>
__global__ void __launch_bounds__(BUCKET_TPB) k_bucket_scan(int *cnt, int n, int nt, int *slow,
                                                            unsigned long long *state, int *ticket,
                                                            uint32_t *status) {
    HFCR_PDL_WAIT();
    __shared__ int cta;
    __shared__ unsigned ws[BUCKET_TPB / 32], base;
    if (threadIdx.x == 0) cta = atomicAdd(ticket, 1);
    __syncthreads();
    constexpr int PER = BUCKET_SCAN / BUCKET_TPB;
    const int i0 = cta * BUCKET_SCAN + threadIdx.x * PER;
    unsigned v[PER], sum = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        v[k] = i0 + k < n ? (unsigned)cnt[i0 + k] : 0u;
        sum += v[k];
    }
    unsigned total;
    unsigned e = cta_scan(sum, ws, total);
    if (threadIdx.x < 32) {
        const unsigned b = lookback(state, cta, total, status);
        if (threadIdx.x == 0) base = b;
    }
    if constexpr (HUBS) {  // meanwhile: the long lists of one CTA of k_bucket_edges
        unsigned cost = 0;
        if (sum > (unsigned)BUCKET_SHORT) {
#pragma unroll
            for (int k = 0; k < PER; ++k)
                if (v[k] > (unsigned)BUCKET_SHORT) cost += bucket_cost(v[k], (unsigned)n / (32 * BUCKET_SM) + 1);
        }
        if (__any_sync(0xffffffffu, cost != 0)) {
            cost = __reduce_add_sync(0xffffffffu, cost);
            if ((threadIdx.x & 31) == 0 && cost > bucket_cost_limit(nt)) *slow = 1;
        }
    }
    __syncthreads();
    e += base;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (i0 + k < n) cnt[i0 + k] = (int)e;
        e += v[k];
        if (i0 + k == n - 1) cnt[n] = (int)e;
    }
}

template <bool HUBS>
__global__ void __launch_bounds__(BUCKET_TPB) k_bucket_fill(const int *tris, int nt, int nv, const int *ptr,
                                                            const typename BucketRank<HUBS>::T *rank, const int *slow, int *bucket) {
    HFCR_PDL_WAIT();
    const int t = blockIdx.x * BUCKET_TPB + threadIdx.x;
    if (t >= nt) return;
    const int v[3] = {tris[3 * t], tris[3 * t + 1], tris[3 * t + 2]};
    const int r[3] = {rank[3 * t], rank[3 * t + 1], rank[3 * t + 2]};
    if (*slow) return;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int a = v[k], b = v[(k + 1) % 3];
        if ((unsigned)a >= (unsigned)nv || (unsigned)b >= (unsigned)nv) a = b = 0;
        bucket[ptr[min(a, b)] + r[k]] = max(a, b);
    }
}

// list[0 .. n) ascending and without repeats, in place; returns the length
__device__ __forceinline__ int sort_unique(int *list, int n) {
    for (int i = 1; i < n; ++i) {
        const int x = list[i];
        int j = i - 1;
        while (j >= 0 && list[j] > x) {
            list[j + 1] = list[j];
            --j;
        }
        list[j + 1] = x;
    }
    int m = 0, last = -1;
    for (int i = 0; i < n; ++i) {
        const int x = list[i];
        if (x != last) list[m++] = x;
        last = x;
    }
    return m;
}

// One warp: src[0 .. n) ascending to tmp, then without repeats to dst (which
// may be src or tmp); returns the length
__device__ __forceinline__ int warp_sort_unique(const int *src, int n, int *tmp, int *dst) {
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int i = lane; i < n; i += 32) {  // an entry's place: the smaller ones, and equal ones before it
        const int x = src[i];
        int r = 0;
#pragma unroll 4
        for (int q = 0; q < n; ++q) {
            const int y = src[q];
            r += y < x || (y == x && q < i);
        }
        tmp[r] = x;
    }
    __syncwarp();
    int m = 0, last = -1;
#pragma unroll 1
    for (int q = 0; q < n; q += 32) {  // never writes past what it has read
        const int y = q + lane < n ? tmp[q + lane] : -1;
        int prev = __shfl_up_sync(0xffffffffu, y, 1);
        if (lane == 0) prev = last;
        const bool keep = q + lane < n && y != prev;
        const unsigned k = __ballot_sync(0xffffffffu, keep);
        if (keep) dst[m + __popc(k & ((1u << lane) - 1u))] = y;
        m += __popc(k);
        last = __shfl_sync(0xffffffffu, y, 31);
        __syncwarp();
    }
    return m;
}

// The CTA: src[0 .. n) ascending and without repeats to dst, through a bitmap
// of bits words (as many passes as its range needs); returns the length
__device__ __forceinline__ int cta_sort_unique(const int *src, int n, int *dst, unsigned *bits, unsigned *ws,
                                               int *range) {
    constexpr int SPAN = 32 * BUCKET_SM;
    if (threadIdx.x == 0) {
        range[0] = 0x7fffffff;
        range[1] = 0;
    }
    __syncthreads();
    int lo = 0x7fffffff, hi = 0;
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += BUCKET_TPB) {
        const int x = src[i];
        lo = min(lo, x);
        hi = max(hi, x);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(range, lo);
        atomicMax(range + 1, hi);
    }
    __syncthreads();
    const int first = range[0] & ~31, last = range[1];
    unsigned m = 0;
    for (long long b = first; b <= last; b += SPAN) {
        const int words = (int)min((last - b) / 32 + 1, (long long)BUCKET_SM);
        for (int i = threadIdx.x; i < words; i += BUCKET_TPB) bits[i] = 0u;
        __syncthreads();
#pragma unroll 4
        for (int i = threadIdx.x; i < n; i += BUCKET_TPB) {
            const unsigned x = (unsigned)src[i] - (unsigned)b;
            if (x < (unsigned)SPAN) atomicOr(bits + (x >> 5), 1u << (x & 31));
        }
        __syncthreads();
        const int per = (words + BUCKET_TPB - 1) / BUCKET_TPB, i0 = min((int)threadIdx.x * per, words);
        const int i1 = min(i0 + per, words);
        unsigned c = 0, total;
        for (int i = i0; i < i1; ++i) c += __popc(bits[i]);
        unsigned at = m + cta_scan(c, ws, total);
        for (int i = i0; i < i1; ++i)
            for (unsigned y = bits[i]; y; y &= y - 1u) dst[at++] = (int)b + 32 * i + __ffs(y) - 1;
        m += total;
        __syncthreads();  // bits and ws are the next pass's
    }
    return (int)m;
}

// The lists of more than BUCKET_SHORT half-edges of one CTA of k_bucket_edges
// (out of line: the ordinary path then keeps its registers)
struct LongLists {
    unsigned at[BUCKET_TPB];         // each vertex's first edge
    uint16_t len[BUCKET_TPB];        // and its number of them
    unsigned char v[BUCKET_TPB];     // the vertices, in any order
    int n, range[2];
};

// all of them sorted: in place in list (the CTA's in shared memory, or null),
// out as scratch; hubs, and the others without it, to spare
__device__ __noinline__ void sort_long_lists(LongLists &l, const int *ptr, int p0, int *list, int *out,
                                             const int *bucket, int *spare, unsigned *ws) {
    for (int x = threadIdx.x >> 5; x < l.n; x += BUCKET_TPB / 32) {
        const int q = l.v[x], l0 = ptr[q], n = ptr[q + 1] - l0;
        if (n > BUCKET_WARP) continue;
        const int m = list ? warp_sort_unique(list + (l0 - p0), n, out + (l0 - p0), list + (l0 - p0))
                           : warp_sort_unique(bucket + l0, n, spare + l0, spare + l0);
        if ((threadIdx.x & 31) == 0) l.len[q] = (uint16_t)m;
    }
    for (int x = 0; x < l.n; ++x) {
        const int q = l.v[x], l0 = ptr[q], n = ptr[q + 1] - l0;
        if (n <= BUCKET_WARP) continue;
        const int m = cta_sort_unique(bucket + l0, n, spare + l0, (unsigned *)out, ws, l.range);
        if (threadIdx.x == 0) l.len[q] = (uint16_t)m;
    }
    __syncthreads();
}

// their edges, vertex q's from its thread's `at` on: to out and owner, or
// straight to edges (list null)
__device__ __noinline__ void put_long_lists(LongLists &l, const int *ptr, int p0, const int *list,
                                            const int *spare, unsigned at, int v0, int *out,
                                            unsigned char *owner, int2 *edges) {
    l.at[threadIdx.x] = at;
    __syncthreads();
    auto put = [&](int q, const int *from, int first, int step) {
        const unsigned to = l.at[q];
        const int m = l.len[q];
#pragma unroll 4
        for (int i = first; i < m; i += step) {
            const int y = from[i];
            if (list) {
                out[to + i] = y;
                owner[to + i] = (unsigned char)q;
            } else {
                edges[to + i] = make_int2(v0 + q, y);
            }
        }
    };
    for (int x = threadIdx.x >> 5; x < l.n; x += BUCKET_TPB / 32) {
        const int q = l.v[x], l0 = ptr[q], n = ptr[q + 1] - l0;
        if (n <= BUCKET_WARP) put(q, list ? list + (l0 - p0) : spare + l0, threadIdx.x & 31, 32);
    }
    for (int x = 0; x < l.n; ++x) {
        const int q = l.v[x], l0 = ptr[q], n = ptr[q + 1] - l0;
        if (n > BUCKET_WARP) put(q, spare + l0, threadIdx.x, BUCKET_TPB);
    }
}

// spare (HUBS): [the half-edges], the sorted lists of more than BUCKET_SHORT
template <bool HUBS>
__global__ void __launch_bounds__(BUCKET_TPB, 6) k_bucket_edges(const int *ptr, int nv, int *bucket, int *spare,
                                                                int2 *edges, int *d_count, const int *slow,
                                                                unsigned long long *state, int *ticket,
                                                                uint32_t *status) {
    HFCR_PDL_WAIT();
    // a void result is not written (edges may be the caller's own buffer)
    const bool is_void = *slow || (*(volatile uint32_t *)status & ST_BAD_INDEX);
    __shared__ int list[BUCKET_SM], out[BUCKET_SM];
    __shared__ unsigned char owner[BUCKET_SM];
    __shared__ LongLists longs[1];  // (no room is taken where nothing uses it)
    __shared__ unsigned ws[BUCKET_TPB / 32], base;
    __shared__ int cta;
    if (threadIdx.x == 0) {
        cta = atomicAdd(ticket, 1);
        if (HUBS) longs->n = 0;
    }
    __syncthreads();
    if (is_void) return;
    const int v0 = cta * BUCKET_TPB, v = v0 + threadIdx.x, ve = min(v0 + BUCKET_TPB, nv);
    const int p0 = ptr[v0], m = ptr[ve] - p0;
    const bool in_sm = m <= BUCKET_SM;
    const int a = v < nv ? ptr[v] - p0 : 0, n = v < nv ? ptr[v + 1] - p0 - a : 0;
    const bool is_long = HUBS && n > BUCKET_SHORT;
    if (is_long) longs->v[atomicAdd(&longs->n, 1)] = (unsigned char)threadIdx.x;
    if (in_sm)
        for (int i = threadIdx.x; i < m; i += BUCKET_TPB) list[i] = bucket[p0 + i];
    __syncthreads();
    int u = 0;
    if (!is_long) u = in_sm ? sort_unique(list + a, n) : sort_unique(bucket + p0 + a, n);
    if (HUBS && longs->n) {
        sort_long_lists(*longs, ptr + v0, p0, in_sm ? list : nullptr, out, bucket, spare, ws);
        if (is_long) u = longs->len[threadIdx.x];
    }
    unsigned total;
    const unsigned at = cta_scan((unsigned)u, ws, total);
    if (threadIdx.x < 32) {
        const unsigned b = lookback(state, cta, total, status);
        if (threadIdx.x == 0) {
            base = b;
            if (ve == nv) *d_count = (int)(b + total);
        }
    }
    if (in_sm) {  // compacted first, then written in order
        if (!is_long)
            for (int i = 0; i < u; ++i) {
                out[at + i] = list[a + i];
                owner[at + i] = (unsigned char)threadIdx.x;
            }
        if (HUBS && longs->n) put_long_lists(*longs, ptr + v0, p0, list, spare, at, v0, out, owner, edges);
        __syncthreads();
        for (int i = threadIdx.x; i < (int)total; i += BUCKET_TPB)
            edges[base + i] = make_int2(v0 + owner[i], out[i]);
    } else {
        __syncthreads();
        if (!is_long)
            for (int i = 0; i < u; ++i) edges[base + at + i] = make_int2(v, bucket[p0 + a + i]);
        if (HUBS && longs->n)
            put_long_lists(*longs, ptr + v0, p0, nullptr, spare, base + at, v0, out, owner, edges);
    }
}

template <typename T>
__device__ __forceinline__ void load3(const T *x, const T *y, const T *z, int i, T *o) {
    o[0] = x[i];
    o[1] = y[i];
    o[2] = z[i];
}

__device__ __forceinline__ float lo_f(float v) { return v; }
__device__ __forceinline__ float hi_f(float v) { return v; }
__device__ __forceinline__ float lo_f(double v) { return __double2float_rd(v); }
__device__ __forceinline__ float hi_f(double v) { return __double2float_ru(v); }

// per-block min/max of the vertex positions (coalesced; they contain every
// face centroid, and float32 approximations suffice: the codes only order
// the leaves)
template <typename T>
__global__ void k_vertex_bounds(const T *x, const T *y, const T *z, int nv, float *part) {
    HFCR_PDL_WAIT();
    float lo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, hi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x) {
        const float c[3] = {(float)x[v], (float)y[v], (float)z[v]};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            lo[k] = fminf(lo[k], c[k]);
            hi[k] = fmaxf(hi[k], c[k]);
        }
    }
    __shared__ float s[6][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        for (int o = 16; o; o >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
        if (lane == 0) { s[k][w] = lo[k]; s[3 + k][w] = hi[k]; }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        int nw = blockDim.x >> 5;
        float v = s[threadIdx.x][0];
        for (int i = 1; i < nw; ++i)
            v = threadIdx.x < 3 ? fminf(v, s[threadIdx.x][i]) : fmaxf(v, s[threadIdx.x][i]);
        part[6 * blockIdx.x + threadIdx.x] = v;
    }
}

// the nb per-block partials folded by one CTA of 256 threads
__global__ void __launch_bounds__(256) k_bounds_final(const float *part, int nb, float *bounds) {
    HFCR_PDL_WAIT();
    float lo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, hi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
    for (int i = threadIdx.x; i < nb; i += blockDim.x)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            lo[k] = fminf(lo[k], part[6 * i + k]);
            hi[k] = fmaxf(hi[k], part[6 * i + 3 + k]);
        }
    __shared__ float sh[6][8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        for (int o = 16; o; o >>= 1) {
            lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
            hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
        }
        if (lane == 0) { sh[k][w] = lo[k]; sh[3 + k][w] = hi[k]; }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int k = threadIdx.x;
        float v = sh[k][0];
        for (int q = 1; q < (int)(blockDim.x >> 5); ++q) v = k < 3 ? fminf(v, sh[k][q]) : fmaxf(v, sh[k][q]);
        bounds[k] = v;
    }
}

__device__ __forceinline__ unsigned spread10(unsigned v) {
    v = (v * 0x00010001u) & 0xFF0000FFu;
    v = (v * 0x00000101u) & 0x0F00F00Fu;
    v = (v * 0x00000011u) & 0xC30C30C3u;
    v = (v * 0x00000005u) & 0x49249249u;
    return v;
}

// Morton code of each face's centroid, quantised to `cells` per axis in the
// scene bounds (cells <= 1024), above it the face's segment
template <typename T>
__global__ void k_morton(const T *x, const T *y, const T *z, int nv, const int *tris, int nt,
                         const float *bounds, const int *segs, int col, int nseg, float cells,
                         unsigned long long *keys, int *vals, uint32_t *st) {
    HFCR_PDL_WAIT();
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    T a[3], b[3], c[3];
    load3(x, y, z, chk(tris[3 * t], nv, st), a);
    load3(x, y, z, chk(tris[3 * t + 1], nv, st), b);
    load3(x, y, z, chk(tris[3 * t + 2], nv, st), c);
    unsigned q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float m = (float)((a[k] + b[k] + c[k]) / (T)3);
        float ext = bounds[3 + k] - bounds[k];
        float u = ext > 0.f ? (m - bounds[k]) / ext : 0.f;
        u = fminf(fmaxf(u * cells, 0.f), cells - 1.f);
        q[k] = (unsigned)u;
    }
    const unsigned long long seg = (unsigned long long)seg_of(segs, col, nseg, t);
    keys[t] = (seg << 30) | (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
    vals[t] = t;
}

// sort key of an edge: (segment of its first vertex, Morton code of its
// midpoint); value = the edge's index
template <typename T>
__global__ void k_edge_order_keys(const int2 *edges, int ne, const T *x, const T *y, const T *z,
                                  int nv, const float *bounds, const int *segs, int col, int nseg,
                                  unsigned long long *keys, int *vals, uint32_t *st) {
    HFCR_PDL_WAIT();
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= ne) return;
    const int2 ed = edges[e];
    const int a = chk(ed.x, nv, st), b = chk(ed.y, nv, st);
    const T pa[3] = {x[a], y[a], z[a]}, pb[3] = {x[b], y[b], z[b]};
    unsigned q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float m = (float)((pa[k] + pb[k]) / (T)2);
        const float ext = bounds[3 + k] - bounds[k];
        float u = ext > 0.f ? (m - bounds[k]) / ext : 0.f;
        u = fminf(fmaxf(u * 1024.f, 0.f), 1023.f);
        q[k] = (unsigned)u;
    }
    const unsigned long long seg = (unsigned long long)seg_of(segs, col, nseg, a);
    keys[e] = (seg << 30) | (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
    vals[e] = e;
}

// common-prefix length of the keys of leaves i and j of one segment (its
// sorted keys start at K); keys made unique by appending the local index
__device__ __forceinline__ int kdelta(const unsigned long long *K, int n, int i, int j) {
    if (j < 0 || j >= n) return -1;
    unsigned long long ki = ((K[i] & 0x3fffffffull) << 32) | (unsigned)i;
    unsigned long long kj = ((K[j] & 0x3fffffffull) << 32) | (unsigned)j;
    return __clzll(ki ^ kj);
}

// Leaves per block of the refit.  A node is local when its leaf range lies
// in one block [REFIT_BLOCK b, REFIT_BLOCK (b + 1)) (its index is an end of
// that range, so the node does too); the others span blocks.
constexpr int REFIT_BITS = 9;
constexpr int REFIT_BLOCK = 1 << REFIT_BITS;

// Karras 2012, one tree per segment: internal node l of the segment whose
// faces start at t0 covers a key range found from the common-prefix lengths
// of its neighbours.  Segment-local node l is stored at t0 + l, leaf c at
// t0 + c (encoded ~(t0 + c)).  Links carry the child's slot and whether the
// parent is local: (parent << 2) | (local << 1) | (1 for the right child),
// parents being below 2^29; roots (l = 0) keep the -1 the caller set.  The
// nodes that span blocks are listed in top[1 ...], their number in top[0]
// (zeroed by the caller).
__global__ void k_karras(const unsigned long long *keys, int n_total, const int *segs, int col,
                         int nseg, float4 *nodes, int *iparent, int *lparent, int *top) {
    HFCR_PDL_WAIT();
    int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= n_total) return;
    const int sgi = seg_of(segs, col, nseg, gi);
    int t0, n;
    seg_range(segs, col, sgi, n_total, t0, n);
    const int i = gi - t0;
    if (i < 0 || i >= n - 1) return;
    const unsigned long long *K = keys + t0;
    int d = (kdelta(K, n, i, i + 1) - kdelta(K, n, i, i - 1)) >= 0 ? 1 : -1;
    int dmin = kdelta(K, n, i, i - d);
    int lmax = 2;
    while (kdelta(K, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
        if (kdelta(K, n, i, i + (l + t) * d) > dmin) l += t;
    int j = i + l * d;
    int dnode = kdelta(K, n, i, j);
    int s = 0, t = l;
    do {
        t = (t + 1) >> 1;
        if (kdelta(K, n, i, i + (s + t) * d) > dnode) s += t;
    } while (t > 1);
    int gamma = i + s * d + min(d, 0);
    int left = (min(i, j) == gamma) ? ~(t0 + gamma) : t0 + gamma;
    int right = (max(i, j) == gamma + 1) ? ~(t0 + gamma + 1) : t0 + gamma + 1;
    nodes[4 * gi + 3] = make_float4(__int_as_float(left), __int_as_float(right), 0.f, 0.f);
    const bool local = ((t0 + i) >> REFIT_BITS) == ((t0 + j) >> REFIT_BITS);
    const int link = (gi << 2) | (local ? 2 : 0);
    if (left < 0) lparent[~left] = link; else iparent[left] = link;
    if (right < 0) lparent[~right] = link | 1; else iparent[right] = link | 1;
    if (!local) top[1 + atomicAdd(top, 1)] = gi;
}

template <typename T>
__device__ __forceinline__ void pack_leaf(void *leaf_tri, int j, const T *a, const T *b,
                                          const T *c, int f);
template <>
__device__ __forceinline__ void pack_leaf<float>(void *leaf_tri, int j, const float *a,
                                                 const float *b, const float *c, int f) {
    float4 *L = (float4 *)leaf_tri + 3 * j;
    L[0] = make_float4(a[0], a[1], a[2], b[0]);
    L[1] = make_float4(b[1], b[2], c[0], c[1]);
    L[2] = make_float4(c[2], __int_as_float(f), 0.f, 0.f);
}
template <>
__device__ __forceinline__ void pack_leaf<double>(void *leaf_tri, int j, const double *a,
                                                  const double *b, const double *c, int f) {
    double2 *L = (double2 *)leaf_tri + 5 * j;
    L[0] = make_double2(a[0], a[1]);
    L[1] = make_double2(a[2], b[0]);
    L[2] = make_double2(b[1], b[2]);
    L[3] = make_double2(c[0], c[1]);
    L[4] = make_double2(c[2], __longlong_as_double((long long)f));
}

// Refit, first kernel: one CTA per block of REFIT_BLOCK leaves, one thread
// per leaf.  The boxes of the block's local nodes are merged in shared
// memory: both children of a local node are carried by threads of this CTA,
// which meet at the node's slot (an arrival counter, block-scope fences);
// the second carries the union upwards, its links read from shared memory.
// Then thread t writes node base + t.  A box whose parent spans blocks goes
// to the parent's child slot in global memory; the slot of a child that
// itself spans blocks is set empty, for the second kernel.  Min and max are
// exact, so the boxes do not depend on the order.
// Bound by the latency of the position gathers, then by some ten shared-
// memory steps; 512 leaves keep four CTAs on an SM.  With arrival counters in
// global memory for every node above a warp's 32 leaves a level cost about
// 2 us (fence, atomic, sibling read).  Both kernels together, against that
// form: 327,680 float32 faces 71 -> 39 us, 262,144 51 -> 34, 1,280 float64
// faces 24 -> 17, 5.06 million in 1,024 trees 503 -> 273.
template <typename T>
__global__ void __launch_bounds__(REFIT_BLOCK) k_refit_block(
    const T *x, const T *y, const T *z, int nv, const int *tris, const int *leaf_face, int n,
    float4 *nodes, const int *iparent, const int *lparent, void *leaf_tri, uint32_t *st) {
    HFCR_PDL_WAIT();
    __shared__ float sb[12][REFIT_BLOCK];  // both child boxes of each local node
    __shared__ int up[REFIT_BLOCK];
    __shared__ unsigned cnt[REFIT_BLOCK];
    const int t = threadIdx.x, base = blockIdx.x * REFIT_BLOCK, j = base + t;
    const bool live = j < n;
    int link = -1;
    float lo[3] = {0.f, 0.f, 0.f}, hi[3] = {0.f, 0.f, 0.f};
    cnt[t] = 0u;
    up[t] = live ? iparent[j] : -1;
    if (live) {
        link = lparent[j];  // -1: the only face of its segment
        const int f = leaf_face[j];
        T a[3], b[3], c[3];
        load3(x, y, z, chk(tris[3 * f], nv, st), a);
        load3(x, y, z, chk(tris[3 * f + 1], nv, st), b);
        load3(x, y, z, chk(tris[3 * f + 2], nv, st), c);
        pack_leaf<T>(leaf_tri, j, a, b, c, f);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            lo[k] = lo_f(fmin(fmin(a[k], b[k]), c[k]));
            hi[k] = hi_f(fmax(fmax(a[k], b[k]), c[k]));
        }
    }
    __syncthreads();
    // bounded by the tree depth (< 64 for unique 62-bit keys); the guard
    // only keeps a corrupted parent array from looping
    for (int guard = 0; guard < 128 && link >= 0 && (link & 2); ++guard) {
        const int q = (link >> 2) - base;
        if ((unsigned)q >= (unsigned)REFIT_BLOCK) {  // unreachable: a local parent is in the block
            atomicOr(st, ST_BAD_INDEX);
            link = -1;
            break;
        }
        const int o = (link & 1) ? 6 : 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            sb[o + k][q] = lo[k];
            sb[o + 3 + k][q] = hi[k];
        }
        __threadfence_block();
        if (atomicAdd(&cnt[q], 1u) == 0u) {
            link = -1;  // the sibling's thread carries on
            break;
        }
        __threadfence_block();
        const volatile float *vs = &sb[0][0] + q;
        const int so = 6 - o;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            lo[k] = fminf(lo[k], vs[(so + k) * REFIT_BLOCK]);
            hi[k] = fmaxf(hi[k], vs[(so + 3 + k) * REFIT_BLOCK]);
        }
        link = up[q];
    }
    if (link >= 0) {
        float2 *s = (float2 *)((float *)(nodes + 4 * (size_t)(link >> 2)) + ((link & 1) ? 6 : 0));
        s[0] = make_float2(lo[0], lo[1]);
        s[1] = make_float2(lo[2], hi[0]);
        s[2] = make_float2(hi[1], hi[2]);
    }
    __syncthreads();
    if (!live) return;
    if (cnt[t] == 2u) {
        float4 *nd = nodes + 4 * (size_t)j;
        nd[0] = make_float4(sb[0][t], sb[1][t], sb[2][t], sb[3][t]);
        nd[1] = make_float4(sb[4][t], sb[5][t], sb[6][t], sb[7][t]);
        nd[2] = make_float4(sb[8][t], sb[9][t], sb[10][t], sb[11][t]);
    } else if (up[t] >= 0) {  // a node that spans blocks (and is not a root)
        const int l = up[t];
        const float inf = __int_as_float(0x7f800000);
        float2 *s = (float2 *)((float *)(nodes + 4 * (size_t)(l >> 2)) + ((l & 1) ? 6 : 0));
        s[0] = make_float2(inf, inf);
        s[1] = make_float2(inf, -inf);
        s[2] = make_float2(-inf, -inf);
    }
}

// *p = min(*p, v) / max(*p, v) of floats by integer atomics: non-negative
// floats order as signed integers, negative ones in reverse as unsigned
__device__ __forceinline__ void red_min(float *p, float v) {
    const int b = __float_as_int(v);
    if (b >= 0) atomicMin((int *)p, b);
    else atomicMax((unsigned *)p, (unsigned)b);
}
__device__ __forceinline__ void red_max(float *p, float v) {
    const int b = __float_as_int(v);
    if (b >= 0) atomicMax((int *)p, b);
    else atomicMin((unsigned *)p, (unsigned)b);
}

// Refit, second kernel: one thread per node that spans blocks.  It carries
// the union of the child boxes it finds (those of local children, written by
// the first kernel) up the tree, widening each ancestor's slot by atomics
// that nothing waits for, and stops where the slot already holds its box:
// whoever widened that slot carries the same bounds on, so every slot ends
// as the union over its leaves.  There are about ten such nodes per block
// boundary, and a step costs one read of the slot instead of a handshake.
__global__ void __launch_bounds__(256) k_refit_top(float4 *nodes, const int *iparent,
                                                   const int *top, int n) {
    HFCR_PDL_WAIT();
    const int nt = min(top[0], n);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nt; i += gridDim.x * blockDim.x) {
        const int node = top[1 + i];
        const float2 *c = (const float2 *)(nodes + 4 * (size_t)node);
        float2 v[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = __ldcg(c + k);
        const float lo[3] = {fminf(v[0].x, v[3].x), fminf(v[0].y, v[3].y), fminf(v[1].x, v[4].x)};
        const float hi[3] = {fmaxf(v[1].y, v[4].y), fmaxf(v[2].x, v[5].x), fmaxf(v[2].y, v[5].y)};
        int link = iparent[node];
        for (int guard = 0; guard < 128 && link >= 0; ++guard) {
            const int p = link >> 2;
            float *s = (float *)(nodes + 4 * (size_t)p) + ((link & 1) ? 6 : 0);
            const float2 a = __ldcg((const float2 *)s), b = __ldcg((const float2 *)s + 1),
                         d = __ldcg((const float2 *)s + 2);
            link = iparent[p];
            bool wider = false;
            if (lo[0] < a.x) { red_min(s, lo[0]); wider = true; }
            if (lo[1] < a.y) { red_min(s + 1, lo[1]); wider = true; }
            if (lo[2] < b.x) { red_min(s + 2, lo[2]); wider = true; }
            if (hi[0] > b.y) { red_max(s + 3, hi[0]); wider = true; }
            if (hi[1] > d.x) { red_max(s + 4, hi[1]); wider = true; }
            if (hi[2] > d.y) { red_max(s + 5, hi[2]); wider = true; }
            if (!wider) break;
        }
    }
}

}  // namespace

void validate_positions(const hfcr_mesh &m, uint32_t *d_status, cudaStream_t s) {
    if (m.n_verts <= 0) return;
    int nb = (m.n_verts + 255) / 256;
    if (m.dtype == HFCR_F32)
        { launch_pdl(k_validate<float>, nb, 256, 0, s, (const float *)m.x, (const float *)m.y,
                                             (const float *)m.z, m.n_verts, d_status); note_launch(); }
    else
        { launch_pdl(k_validate<double>, nb, 256, 0, s, (const double *)m.x, (const double *)m.y,
                                              (const double *)m.z, m.n_verts, d_status); note_launch(); }
}

void validate_pair(const hfcr_mesh &A, const hfcr_mesh &B, uint32_t *d_status, cudaStream_t s) {
    if (A.dtype != B.dtype) {
        validate_positions(A, d_status, s);
        validate_positions(B, d_status, s);
        return;
    }
    const int nA = A.n_verts > 0 ? A.n_verts : 0, nB = B.n_verts > 0 ? B.n_verts : 0;
    if (nA + nB <= 0) return;
    const int nb = (nA + nB + 255) / 256;
    if (A.dtype == HFCR_F32)
        { launch_pdl(k_validate_pair<float>, nb, 256, 0, s, (const float *)A.x, (const float *)A.y,
                     (const float *)A.z, nA, (const float *)B.x, (const float *)B.y,
                     (const float *)B.z, nB, d_status); note_launch(); }
    else
        { launch_pdl(k_validate_pair<double>, nb, 256, 0, s, (const double *)A.x,
                     (const double *)A.y, (const double *)A.z, nA, (const double *)B.x,
                     (const double *)B.y, (const double *)B.z, nB, d_status); note_launch(); }
}

void build_edges_sorted(const int *tris, int n_tris, int n_verts, int *edges_out, int *d_count,
                 unsigned long long *keys, unsigned long long *keys_alt, unsigned *flags,
                 SortTemp &t, uint32_t *d_status, cudaStream_t s) {
    int n = 3 * n_tris;
    if (n == 0) {
        cudaMemsetAsync(d_count, 0, sizeof(int), s);
        return;
    }
    int vb = bits_for(n_verts > 1 ? n_verts : 2);
    { launch_pdl(k_edge_keys, (n_tris + 255) / 256, 256, 0, s, tris, n_tris, vb, keys, d_status,
                 n_verts); note_launch(); }
    bool flip = radix_sort_u64(keys, nullptr, keys_alt, nullptr, n, 2 * vb, t, s);
    unsigned long long *sorted = flip ? keys_alt : keys;
    { launch_pdl(k_unique_flags, (n + 255) / 256, 256, 0, s, sorted, n, flags); note_launch(); }
    scan_flags_dev(flags, nullptr, n, d_count, t, s);
    { launch_pdl(k_write_edges, (n + 255) / 256, 256, 0, s, sorted, flags, n, vb,
                 edges_out); note_launch(); }
}

size_t bucket_words(int n_verts) {
    // counts, both tickets, then both scans' states (8 B each)
    const size_t c = (size_t)n_verts + 4;
    const size_t st = ((size_t)n_verts + BUCKET_SCAN - 1) / BUCKET_SCAN + ((size_t)n_verts + BUCKET_TPB - 1) / BUCKET_TPB;
    return ((c + 1) & ~(size_t)1) + 2 * st;
}

template <bool HUBS>
static void bucket_edges(const int *tris, int n_tris, int n_verts, int *edges_out, int *d_count, int *d_slow,
                         unsigned long long *keys, unsigned long long *keys_alt, int *words, uint32_t *d_status,
                         cudaStream_t s) {
    typedef typename BucketRank<HUBS>::T Rank;
    int *bucket = (int *)keys, *spare = bucket + 3 * (size_t)n_tris;  // [3 n_tris] each
    Rank *rank = (Rank *)keys_alt;                                    // [3 n_tris]
    int *cnt = words, *tickets = words + n_verts + 1;
    const int nscan = (n_verts + BUCKET_SCAN - 1) / BUCKET_SCAN;
    unsigned long long *state = (unsigned long long *)(words + (((size_t)n_verts + 4 + 1) & ~(size_t)1));
    cudaMemsetAsync(words, 0, sizeof(int) * bucket_words(n_verts), s);
    const int nb = (n_tris + BUCKET_TPB - 1) / BUCKET_TPB, vb = (n_verts + BUCKET_TPB - 1) / BUCKET_TPB;
    { launch_pdl(k_bucket_count<HUBS>, nb, BUCKET_TPB, 0, s, tris, n_tris, n_verts, cnt, rank, d_slow,
                 d_status); note_launch(); }
    { launch_pdl(k_bucket_scan<HUBS>, nscan, BUCKET_TPB, 0, s, cnt, n_verts, n_tris, d_slow, state, tickets,
                 d_status); note_launch(); }
    { launch_pdl(k_bucket_fill<HUBS>, nb, BUCKET_TPB, 0, s, tris, n_tris, n_verts, (const int *)cnt,
                 (const Rank *)rank, (const int *)d_slow, bucket); note_launch(); }
    { launch_pdl(k_bucket_edges<HUBS>, vb, BUCKET_TPB, 0, s, (const int *)cnt, n_verts, bucket, spare,
                 (int2 *)edges_out, d_count, (const int *)d_slow, state + nscan, tickets + 1, d_status);
      note_launch(); }
}

bool bucket_hubs_first(int n_tris) { return n_tris <= BUCKET_HUBS_TRIS; }

// The buckets pass over every vertex id (some 40 us a million), the sort over the
// half-edges (by ranks up to RANK_MAX of them, 50 us; 85 us and 0.27 a thousand
// triangles above): a short list over many ids is the sort's.  1,000 triangles
// of 2,000,000 ids 107 us by buckets and 50 by the sort, 100,000 of 10,000,000
// 427 and 108; 20,000 of 1,000,000 79 and 89.
bool bucket_worth(int n_tris, int n_verts) {
    const long long most = 3ll * n_tris <= RANK_MAX ? 300000 : 1000000 + 5ll * n_tris;
    return n_verts <= most;
}

void build_edges(const int *tris, int n_tris, int n_verts, bool hubs, int *edges_out, int *d_count, int *d_slow,
                 unsigned long long *keys, unsigned long long *keys_alt, int *words, uint32_t *d_status,
                 cudaStream_t s) {
    (hubs ? bucket_edges<true> : bucket_edges<false>)(tris, n_tris, n_verts, edges_out, d_count, d_slow, keys,
                                                      keys_alt, words, d_status, s);
}

void check_segments(const int *segs, int nseg, const hfcr_mesh &A, const hfcr_mesh &B,
                    uint32_t *d_status, cudaStream_t s) {
    { launch_pdl(k_check_segs, (nseg + 1 + 127) / 128, 128, 0, s, segs, nseg, A.n_verts, A.n_tris,
                 B.n_verts,
                                                        B.n_tris, d_status); note_launch(); }
}

void bvh_build(Bvh &b, const hfcr_mesh &m, const int *segs, int col, int nseg, SortTemp &t,
               uint32_t *d_status, cudaStream_t s) {
    int nv = m.n_verts;
    int n = m.n_tris;
    b.n = n;
    b.dtype = m.dtype;
    b.segs = segs;
    b.col = col;
    b.nseg = nseg;
    if (n <= 0) return;
    int nb = (n + 255) / 256;
    // one mesh: 8 bits per axis (24-bit codes, three radix passes; at the
    // face counts here a cell holds about one or two centroids, and equal
    // codes are ordered by face index); a batch: 10 bits per axis below the
    // segment number, each pair's faces sorted by their own CTA
    const bool single = nseg <= 1;
    const float cells = single ? 256.f : 1024.f;
    const int kbits = single ? 24 : 30 + bits_for(nseg + 1);
    // an odd pass count of the one-mesh sort starts from the spare buffers,
    // so that the sorted keys and faces end in the tree's own
    const bool odd = single && (((kbits + 7) / 8) & 1);
    unsigned long long *kin = odd ? b.keys_alt : b.keys, *kout = odd ? b.keys : b.keys_alt;
    int *vin = odd ? b.vals_alt : b.leaf_face, *vout = odd ? b.leaf_face : b.vals_alt;
    int vbk = (nv + 255) / 256;
    if (vbk > 1024) vbk = 1024;
    if (vbk < 1) vbk = 1;
    if (m.dtype == HFCR_F32) {
        const float *x = (const float *)m.x, *y = (const float *)m.y, *z = (const float *)m.z;
        { launch_pdl(k_vertex_bounds<float>, vbk, 256, 0, s, x, y, z, nv,
                     b.bounds_part); note_launch(); }
        { launch_pdl(k_bounds_final, 1, 256, 0, s, b.bounds_part, vbk, b.bounds); note_launch(); }
        { launch_pdl(k_morton<float>, nb, 256, 0, s, x, y, z, nv, m.tris, n, b.bounds, segs, col,
                     nseg, cells, kin, vin, d_status); note_launch(); }
    } else {
        const double *x = (const double *)m.x, *y = (const double *)m.y, *z = (const double *)m.z;
        { launch_pdl(k_vertex_bounds<double>, vbk, 256, 0, s, x, y, z, nv,
                     b.bounds_part); note_launch(); }
        { launch_pdl(k_bounds_final, 1, 256, 0, s, b.bounds_part, vbk, b.bounds); note_launch(); }
        { launch_pdl(k_morton<double>, nb, 256, 0, s, x, y, z, nv, m.tris, n, b.bounds, segs, col,
                     nseg, cells, kin, vin, d_status); note_launch(); }
    }
    // a batch sorts each pair's faces in its own CTA (the segment bits above
    // the 30 Morton bits are constant within a pair); one mesh globally
    bool flip = !single
                    ? radix_sort_u64v_segments(b.keys, b.leaf_face, b.keys_alt, b.vals_alt, n,
                                               kbits, segs, col, nseg, 30, b.d_rest, t, s)
                    : radix_sort_u64(kin, vin, kout, vout, n, kbits, t, s) != (kin == b.keys_alt);
    if (flip) {
        cudaMemcpyAsync(b.keys, b.keys_alt, sizeof(unsigned long long) * n, cudaMemcpyDeviceToDevice, s);
        cudaMemcpyAsync(b.leaf_face, b.vals_alt, sizeof(int) * n, cudaMemcpyDeviceToDevice, s);
    }
    // roots and leaves of one-face segments keep parent -1 (and so does
    // whatever a malformed segment table leaves out of every tree)
    cudaMemsetAsync(b.parent, 0xff, sizeof(int) * n, s);
    cudaMemsetAsync(b.parent + b.cap, 0xff, sizeof(int) * n, s);
    cudaMemsetAsync(b.top, 0, sizeof(int), s);
    { launch_pdl(k_karras, nb, 256, 0, s, b.keys, n, segs, col, nseg, b.nodes, b.parent,
                 b.parent + b.cap, b.top); note_launch(); }
}

void edge_order(const int *edges, int ne, const hfcr_mesh &m, const int *segs, int col, int nseg,
                int *order, int *order_alt, unsigned long long *keys, unsigned long long *keys_alt,
                float *bounds_part, float *bounds, SortTemp &t, uint32_t *d_status, cudaStream_t s) {
    if (ne <= 0 || m.n_verts <= 0) return;
    const int nv = m.n_verts, nb = (ne + 255) / 256;
    int vbk = (nv + 255) / 256;
    if (vbk > 1024) vbk = 1024;
    if (m.dtype == HFCR_F32) {
        const float *x = (const float *)m.x, *y = (const float *)m.y, *z = (const float *)m.z;
        { launch_pdl(k_vertex_bounds<float>, vbk, 256, 0, s, x, y, z, nv,
                     bounds_part); note_launch(); }
        { launch_pdl(k_bounds_final, 1, 256, 0, s, bounds_part, vbk, bounds); note_launch(); }
        { launch_pdl(k_edge_order_keys<float>, nb, 256, 0, s, (const int2 *)edges, ne, x, y, z,
                     nv, bounds, segs,
                                                    col, nseg, keys, order, d_status); note_launch(); }
    } else {
        const double *x = (const double *)m.x, *y = (const double *)m.y, *z = (const double *)m.z;
        { launch_pdl(k_vertex_bounds<double>, vbk, 256, 0, s, x, y, z, nv,
                     bounds_part); note_launch(); }
        { launch_pdl(k_bounds_final, 1, 256, 0, s, bounds_part, vbk, bounds); note_launch(); }
        { launch_pdl(k_edge_order_keys<double>, nb, 256, 0, s, (const int2 *)edges, ne, x, y, z,
                     nv, bounds, segs,
                                                     col, nseg, keys, order, d_status); note_launch(); }
    }
    if (radix_sort_u64(keys, order, keys_alt, order_alt, ne, 30 + bits_for(nseg + 1), t, s))
        cudaMemcpyAsync(order, order_alt, sizeof(int) * (size_t)ne, cudaMemcpyDeviceToDevice, s);
}

void bvh_refit(Bvh &b, const hfcr_mesh &m, uint32_t *d_status, cudaStream_t s) {
    const int n = b.n;
    if (n <= 0) return;
    const int nb = (n + REFIT_BLOCK - 1) / REFIT_BLOCK;
    if (m.dtype == HFCR_F32)
        { launch_pdl(k_refit_block<float>, nb, REFIT_BLOCK, 0, s, (const float *)m.x,
                     (const float *)m.y, (const float *)m.z, m.n_verts, m.tris, b.leaf_face, n,
                     b.nodes, b.parent, b.parent + b.cap, b.leaf_tri, d_status); note_launch(); }
    else
        { launch_pdl(k_refit_block<double>, nb, REFIT_BLOCK, 0, s, (const double *)m.x,
                     (const double *)m.y, (const double *)m.z, m.n_verts, m.tris, b.leaf_face, n,
                     b.nodes, b.parent, b.parent + b.cap, b.leaf_tri, d_status); note_launch(); }
    if (nb == 1) return;  // every node is local
    int gt = (16 * nb + 255) / 256;  // about ten spanning nodes per block boundary
    if (gt > 1216) gt = 1216;
    { launch_pdl(k_refit_top, gt, 256, 0, s, b.nodes, b.parent, b.top, n); note_launch(); }
}

}  // namespace hfcr
