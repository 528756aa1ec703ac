// Constraint assembly and the global displacement minimizer (Sec. 4).
//
// Stencil s = {x0; x1, x2, x3} gives the row of grad(D) (Eq. 2): +n^T at x0
// and -n^T/3 at x1, x2, x3, n the unit normal of the face on the
// pre-response positions; D = n . (x0 - (x1 + x2 + x3)/3) (Eq. 1) and the
// right-hand side of Eq. 8 is b = D - d.  The system
// grad(D) M^-1 grad(D)^T lambda = b (Eq. 7 / Eq. 8) is solved matrix-free:
//   u = M^-1 grad(D)^T p   (per touched vertex: a fixed-order sum over the
//                           vertex's stencil entries, a CSR built by a
//                           stable sort, hence deterministic)
//   q = grad(D) u          (per stencil: gather of four vertices).
// Displacement x' - x = -M^-1 grad(D)^T lambda (Eq. 5).
//
// The matrix is block-diagonal by impact zone (stencils that share a vertex:
// connected components by min-label hooking or a lock-free union-find, both
// giving each zone its smallest stencil as label); every zone is solved on
// its own.  The response setup (vertex CSR, zones, zone-ordered rows and
// CSR, preconditioner groups) runs in one cooperative launch (k_setup), or
// as a sequence of kernels.
// MIXED: per zone (a thread group sized to the zone: one warp up to 32
// stencils, a 256-thread half CTA up to 255, a 512-thread CTA up to 1,023,
// a 512-thread CTA with all of an SM's shared memory above, an 8-CTA
// cluster beyond that; staged in shared memory), conjugate gradients in float32 on
// float32 normals, preconditioned by the inverses of the blocks of rows that
// share x0, solve for a correction of lambda; the zone's residual
// b - A lambda is recomputed in float64 with the float64 normals after every
// run (iterative refinement), until |r_zone| <= rel_tol |b_zone|.
// FP64: conjugate gradients in float64 on the whole system.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cooperative_groups.h>

#include "internal.h"
#include "sortdev.cuh"

namespace hfcr {

namespace {

constexpr int CG_THREADS = 1024;
constexpr int BIG_ZONE_THREADS = 512;  // threads of the solver of the zones of ZONE_BIG rows or more

// Loads of data written earlier in the same launch: plain where only the
// loading CTA wrote it (PlainLd), through L2 where another CTA may have
// (L2Ld), never through a possibly stale L1 line.
struct PlainLd {
    static constexpr bool L2 = false;
    template <class T> __device__ static T ld(const T *p) { return *p; }
};
struct L2Ld {
    static constexpr bool L2 = true;
    template <class T> __device__ static T ld(const T *p) { return __ldcg(p); }
};

template <class G>
__device__ __forceinline__ double4_32a ld_n64(const double4_32a *p) {
    if (!G::L2) return *p;
    const double2 lo = __ldcg((const double2 *)p), hi = __ldcg((const double2 *)p + 1);
    double4_32a r;
    r.x = lo.x; r.y = lo.y; r.z = hi.x; r.w = hi.y;
    return r;
}

constexpr int RES_BLOCKS = 512;

__device__ __forceinline__ int chk(int i, int n, uint32_t *st) {
    if ((unsigned)i < (unsigned)n) return i;
    atomicOr(st, ST_BAD_INDEX);
    return 0;
}

template <typename T>
__device__ __forceinline__ double ldd(const void *p, int i) {
    return (double)((const T *)p)[i];
}

__device__ __forceinline__ void ld_pos(const hfcr_mesh &m, int i, double *o) {
    if (m.dtype == HFCR_F32) {
        o[0] = ldd<float>(m.x, i); o[1] = ldd<float>(m.y, i); o[2] = ldd<float>(m.z, i);
    } else {
        o[0] = ldd<double>(m.x, i); o[1] = ldd<double>(m.y, i); o[2] = ldd<double>(m.z, i);
    }
}

// the largest of a non-negative double over the warp into *dst: the bit
// patterns of non-negative doubles order like the unsigned integers
__device__ __forceinline__ void warp_max_to(double v, unsigned long long *dst) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0 && v > 0.0) atomicMax(dst, (unsigned long long)__double_as_longlong(v));
}

// row s of the constraints (Eq. 1, Eq. 2) and its right-hand side (Eq. 8);
// returns |b_s|
__device__ __forceinline__ double assemble_row(const hfcr_mesh &A, const hfcr_mesh &B,
                                               const hfcr_stencil *st, int s, double d, int4 *ids,
                                               double4_32a *n64, float4 *n32, double *b,
                                               uint32_t *status) {
    hfcr_stencil S = st[s];
    const int nA = A.n_verts;
    const hfcr_mesh &E = S.dir ? B : A;  // mesh of x0
    const hfcr_mesh &F = S.dir ? A : B;  // mesh of the face
    if (S.dir > 1u) atomicOr(status, ST_BAD_INDEX);
    int x0 = chk((int)S.x0, E.n_verts, status);
    int f = chk((int)S.face, F.n_tris, status);
    int v1 = chk(F.tris[3 * f], F.n_verts, status), v2 = chk(F.tris[3 * f + 1], F.n_verts, status),
        v3 = chk(F.tris[3 * f + 2], F.n_verts, status);
    double p0[3], p1[3], p2[3], p3[3];
    ld_pos(E, x0, p0);
    ld_pos(F, v1, p1);
    ld_pos(F, v2, p2);
    ld_pos(F, v3, p3);
    double e1[3] = {p2[0] - p1[0], p2[1] - p1[1], p2[2] - p1[2]};
    double e2[3] = {p3[0] - p1[0], p3[1] - p1[1], p3[2] - p1[2]};
    double n[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2],
                   e1[0] * e2[1] - e1[1] * e2[0]};
    double nn = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
    double D = 0.0;
    if (nn > 0.0) {
        n[0] /= nn; n[1] /= nn; n[2] /= nn;
        double c[3];
        for (int q = 0; q < 3; ++q) c[q] = p0[q] - (p1[q] + p2[q] + p3[q]) / 3.0;
        D = n[0] * c[0] + n[1] * c[1] + n[2] * c[2];
    } else {
        n[0] = n[1] = n[2] = 0.0;  // zero-area face: an empty row, b = 0 (only from caller input)
    }
    int o = S.dir ? 0 : nA;  // offset of the face mesh in the global numbering
    int g0 = S.dir ? nA + x0 : x0;
    ids[s] = make_int4(g0, o + v1, o + v2, o + v3);
    n64[s] = make_double4_32a(n[0], n[1], n[2], 0.0);
    n32[s] = make_float4((float)n[0], (float)n[1], (float)n[2], 0.f);
    const double bs = nn > 0.0 ? D - d : 0.0;
    b[s] = bs;
    return fabs(bs);
}

// the rows, and the largest |b| of the call into *max_rhs
__global__ void k_assemble(hfcr_mesh A, hfcr_mesh B, const hfcr_stencil *st, const int *d_k,
                           int cap, double d, int4 *ids, double4_32a *n64, float4 *n32, double *b,
                           unsigned long long *max_rhs, uint32_t *status) {
    HFCR_PDL_WAIT();
    const int k = min(*d_k, cap);
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const double mb = s < k ? assemble_row(A, B, st, s, d, ids, n64, n32, b, status) : 0.0;
    warp_max_to(mb, max_rhs);
}

__global__ void k_csr_entries(const int4 *ids, const int *d_k, int cap, unsigned *key, int *val) {
    HFCR_PDL_WAIT();
    int k = min(*d_k, cap);
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 4 * k) return;
    int s = i >> 2, role = i & 3;
    key[i] = (unsigned)((const int *)ids)[4 * s + role];
    val[i] = i;  // s * 4 + role
}

__global__ void k_csr_flags(const unsigned *key, const int *d_k, int cap, unsigned *flag,
                            int *d_n4) {
    HFCR_PDL_WAIT();
    int n = 4 * min(*d_k, cap);
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) *d_n4 = n;
    if (i < n) flag[i] = (i == 0 || key[i] != key[i - 1]) ? 1u : 0u;
}

__global__ void k_csr_build(const unsigned *key, const int *val, const unsigned *excl,
                            const int *d_k, int cap, int nA, const float *wA, const float *wB,
                            int4 *vidx, int *seg, int *gvert, float *winv) {
    HFCR_PDL_WAIT();
    int n = 4 * min(*d_k, cap);
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned f = (i == 0 || key[i] != key[i - 1]) ? 1u : 0u;
    int j = (int)(excl[i] + f) - 1;
    ((int *)vidx)[val[i]] = j;
    if (f) {
        int g = (int)key[i];
        seg[j] = i;
        gvert[j] = g;
        const float *w = g < nA ? wA : wB;
        int lv = g < nA ? g : g - nA;
        winv[j] = w ? w[lv] : 1.0f;
    }
    if (i == n - 1) seg[j + 1] = n;
}

template <typename T>
__device__ __forceinline__ T block_sum(T v, T *sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        T x = lane < (int)(blockDim.x >> 5) ? sh[lane] : (T)0;
#pragma unroll
        for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) sh[32] = x;
    }
    __syncthreads();
    return sh[32];
}

template <typename T>
struct NrmT;
template <>
struct NrmT<float> { typedef float4 type; };
template <>
struct NrmT<double> { typedef double4_32a type; };

// Conjugate gradients on A x = rhs, A = J M^-1 J^T, by one CTA.
// mode 0 (MIXED inner run): rhs = r64, skipped when ctl[0] (done) is set,
//   on exit lam += x.  mode 1 (FP64): rhs = b, on exit lam = x.
// ctl[0] done flag, ctl[1] total iterations, ctl[2] inner runs.
template <typename T>
__global__ void __launch_bounds__(CG_THREADS) k_cg(
    int mode, const int *d_k, const int *d_U, const int *seg, const int *cval, const float *winv,
    const typename NrmT<T>::type *nrm, const int4 *vidx, const double *rhs64, double *lam, T *x,
    T *r, T *p, T *q, T *u, int maxit, double tol, int *ctl) {
    HFCR_PDL_WAIT();
    __shared__ T sh[33];
    if (mode == 0 && ctl[0]) return;
    const int k = *d_k, U = *d_U, tid = threadIdx.x;
    T rr_loc = 0;
    for (int s = tid; s < k; s += CG_THREADS) {
        T v = (T)rhs64[s];
        r[s] = v;
        p[s] = v;
        x[s] = 0;
        rr_loc += v * v;
    }
    T rr = block_sum(rr_loc, sh);
    const T rr0 = rr;
    const T third = (T)1 / (T)3;
    const T stop = (T)(tol * tol) * rr0;
    int it = 0;
    while (it < maxit && rr > stop && rr > (T)0) {
        // u = M^-1 J^T p
        for (int j = tid; j < U; j += CG_THREADS) {
            T a0 = 0, a1 = 0, a2 = 0;
            for (int e = seg[j]; e < seg[j + 1]; ++e) {
                int v = cval[e];
                int s = v >> 2;
                T c = (v & 3) ? -third : (T)1;
                T ps = c * p[s];
                typename NrmT<T>::type n = nrm[s];
                a0 += ps * (T)n.x;
                a1 += ps * (T)n.y;
                a2 += ps * (T)n.z;
            }
            T w = (T)winv[j];
            u[3 * j] = w * a0;
            u[3 * j + 1] = w * a1;
            u[3 * j + 2] = w * a2;
        }
        __syncthreads();
        // q = J u, pq = p . q
        T pq_loc = 0;
        for (int s = tid; s < k; s += CG_THREADS) {
            int4 vi = vidx[s];
            typename NrmT<T>::type n = nrm[s];
            T d0 = u[3 * vi.x] - (u[3 * vi.y] + u[3 * vi.z] + u[3 * vi.w]) * third;
            T d1 = u[3 * vi.x + 1] - (u[3 * vi.y + 1] + u[3 * vi.z + 1] + u[3 * vi.w + 1]) * third;
            T d2 = u[3 * vi.x + 2] - (u[3 * vi.y + 2] + u[3 * vi.z + 2] + u[3 * vi.w + 2]) * third;
            T qs = (T)n.x * d0 + (T)n.y * d1 + (T)n.z * d2;
            q[s] = qs;
            pq_loc += p[s] * qs;
        }
        T pq = block_sum(pq_loc, sh);
        if (!(pq > (T)0)) break;  // breakdown: A is singular on p
        T alpha = rr / pq;
        T rn_loc = 0;
        for (int s = tid; s < k; s += CG_THREADS) {
            x[s] += alpha * p[s];
            T rs = r[s] - alpha * q[s];
            r[s] = rs;
            rn_loc += rs * rs;
        }
        T rn = block_sum(rn_loc, sh);
        T beta = rn / rr;
        rr = rn;
        for (int s = tid; s < k; s += CG_THREADS) p[s] = r[s] + beta * p[s];
        __syncthreads();
        ++it;
    }
    for (int s = tid; s < k; s += CG_THREADS) {
        if (mode == 0) lam[s] += (double)x[s];
        else lam[s] = (double)x[s];
    }
    if (tid == 0) {
        ctl[1] += it;
        ctl[2] += 1;
    }
}

// ---------------------------------------------------------------------------
// float32 CG of the mixed solver, one CTA, single reduction per iteration
// (Chronopoulos-Gear form: s = A p is carried by a recurrence, so each
// iteration needs one product w = A r and one fused reduction of (r, r) and
// (w, r)).  Everything the iteration touches is staged in shared memory
// when it fits (64 k + 20 U bytes, k stencils, U touched vertices);
// otherwise the same loop runs on global scratch.
// ---------------------------------------------------------------------------

constexpr int FAST_SMEM = 231424;  // 226 KB dynamic (+256 B static) under the 227 KB per-CTA limit
constexpr int ZONE_MID = 256;   // zones with at least this many stencils get all 512 threads
constexpr int ZONE_PAIR_SMEM = 112 * 1024;  // k_cg_zone_pair: 2 CTAs per SM, 56 KB per half
constexpr int ZONE_BIG = 1024;  // zones with at least this many stencils get a CTA of their own

// Index types of a view: the global-memory path reads the int arrays as
// they are; the zone staged in shared memory holds zone-local indices in
// 16 bits (a staged zone has fewer than 2^16 touched vertices and CSR
// entries, since shared memory holds at most 227 KB)
__device__ __forceinline__ int4 as_int4(const int4 &v) { return v; }
__device__ __forceinline__ int4 as_int4(const ushort4 &v) { return make_int4(v.x, v.y, v.z, v.w); }

template <typename VI, typename IX>
struct CgViewT {
    float *r, *p, *x, *sv, *w;   // [k]
    float *z;                    // [k] preconditioned residual P^-1 r
    const float4 *pinv;          // [k] row of its group's inverse block (up to 4 columns)
    const int *gst;              // [G + 1] first row of each group (row offsets relative to the zone)
    int G = 0;                   // groups in the zone
    int goff = 0;                // subtracted from gst values (global path)
    float4 *u;                   // [U] M^-1 J^T r per touched vertex (w unused)
    const float4 *n4;            // [k] unit normals (float32)
    const VI *vidx;              // [k]
    const IX *seg;               // [U + 1]
    const IX *cval;              // [4 k]
    const float *winv;           // [U]
    int voff = 0, coff = 0, eoff = 0;  // subtracted from vidx, cval and seg values (global path)
    // the large zones' preconditioner (null bperm: the groups' inverse rows):
    // blocks of rows sharing x0 or a face; place q of the block order holds
    // row bperm[q], its block starts at place binfo[q] >> 5 and has
    // binfo[q] & 31 rows, and binv + 16 q holds its row of the block's
    // inverse (columns in block order)
    const uint16_t *bperm = nullptr;
    const int *binfo = nullptr;
    const float *binv = nullptr;
    __device__ __forceinline__ float3 nrm(int s) const {
        float4 v = n4[s];
        return make_float3(v.x, v.y, v.z);
    }
};
typedef CgViewT<int4, int> CgView;                // global memory
typedef CgViewT<ushort4, uint16_t> CgViewS;       // staged in shared memory

// deterministic block reduction of three sums with a single barrier: warp
// partials go to red[3 * warp]; after the barrier every warp loads the
// partials lane-parallel, folds them with the same shuffle tree and takes
// lane 0's result (lanes of a butterfly may differ in the last bit; lane
// 0's value is the same in every warp), so all threads get identical sums
__device__ __forceinline__ void block_sum3(float a, float b, float c, float *red, float &sa,
                                           float &sb_, float &sc) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) {
        red[3 * w] = a;
        red[3 * w + 1] = b;
        red[3 * w + 2] = c;
    }
    __syncthreads();
    const int nw = blockDim.x >> 5;
    float x = lane < nw ? red[3 * lane] : 0.f;
    float y = lane < nw ? red[3 * lane + 1] : 0.f;
    float q = lane < nw ? red[3 * lane + 2] : 0.f;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
        q += __shfl_xor_sync(0xffffffffu, q, o);
    }
    sa = __shfl_sync(0xffffffffu, x, 0);
    sb_ = __shfl_sync(0xffffffffu, y, 0);
    sc = __shfl_sync(0xffffffffu, q, 0);
}

// sum over the block, identical in every thread: each warp folds its values
// with a butterfly and keeps lane 0's result, and every warp folds the warps'
// results with the same butterfly
__device__ __forceinline__ double block_sum_uniform(double x, double *redd) {
#pragma unroll
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    x = __shfl_sync(0xffffffffu, x, 0);
    if ((threadIdx.x & 31) == 0) redd[threadIdx.x >> 5] = x;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    double s = lane < (int)(blockDim.x >> 5) ? redd[lane] : 0.0;
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __syncthreads();
    return s;
}

// a, b, c summed over the warp by halving (six shuffles instead of fifteen):
// the lanes 8 k .. 8 k + 7 end with sum k (k < 3)
__device__ __forceinline__ float warp_halve3(float a, float b, float c) {
    const int lane = threadIdx.x & 31;
    const bool h = lane & 16, q = lane & 8;
    const float x = (h ? c : a) + __shfl_xor_sync(0xffffffffu, h ? a : c, 16);
    const float y = (h ? 0.f : b) + __shfl_xor_sync(0xffffffffu, h ? b : 0.f, 16);
    float t = (q ? y : x) + __shfl_xor_sync(0xffffffffu, q ? x : y, 8);
#pragma unroll
    for (int o = 4; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}
// the same over NW warps (8 or 16): each warp's sums to scr[4 w + k], the
// group's barrier, then every warp folds them alike
template <int NW, class F>
__device__ __forceinline__ void group_halve3(float a, float b, float c, float *scr, int w, F sync, float &sa,
                                             float &sb, float &sc) {
    const int lane = threadIdx.x & 31;
    float t = warp_halve3(a, b, c);
    if ((lane & 7) == 0) scr[4 * w + (lane >> 3)] = t;
    sync();
    t = scr[4 * (lane & 7) + (lane >> 3)];
    if (NW == 16) t += scr[4 * ((lane & 7) + 8) + (lane >> 3)];
#pragma unroll
    for (int o = 4; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    sa = __shfl_sync(0xffffffffu, t, 0);
    sb = __shfl_sync(0xffffffffu, t, 8);
    sc = __shfl_sync(0xffffffffu, t, 16);
}

// The thread group that solves one zone: a whole CTA (CtaGroup) or one
// warp (WarpGroup, for small zones; barriers are __syncwarp and every
// reduction stays in shuffles).  Sums are identical in every lane.
struct CtaGroup {
    static constexpr int SIZE = 512;  // of the solvers by rows
    __device__ static void sum3h(float a, float b, float c, float *scr, float &sa, float &sb, float &sc) {
        group_halve3<16>(a, b, c, scr, threadIdx.x >> 5, [] { __syncthreads(); }, sa, sb, sc);
    }
    __device__ static int rank() { return threadIdx.x; }
    __device__ static int size() { return blockDim.x; }
    __device__ static void sync() { __syncthreads(); }
    __device__ static void sum3(float a, float b, float c, float *red, float &sa, float &sb,
                                float &sc) {
        block_sum3(a, b, c, red, sa, sb, sc);
    }
    __device__ static double sum(double x, double *redd) { return block_sum_uniform(x, redd); }
};

struct WarpGroup {
    static constexpr int SIZE = 32;
    __device__ static void sum3h(float a, float b, float c, float *, float &sa, float &sb, float &sc) {
        const float t = warp_halve3(a, b, c);
        sa = __shfl_sync(0xffffffffu, t, 0);
        sb = __shfl_sync(0xffffffffu, t, 8);
        sc = __shfl_sync(0xffffffffu, t, 16);
    }
    __device__ static int rank() { return threadIdx.x & 31; }
    __device__ static int size() { return 32; }
    __device__ static void sync() { __syncwarp(); }
    __device__ static void sum3(float a, float b, float c, float *, float &sa, float &sb, float &sc) {
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
            c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        sa = __shfl_sync(0xffffffffu, a, 0);
        sb = __shfl_sync(0xffffffffu, b, 0);
        sc = __shfl_sync(0xffffffffu, c, 0);
    }
    __device__ static double sum(double x, double *) {
#pragma unroll
        for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        return __shfl_sync(0xffffffffu, x, 0);
    }
};

// One 256-thread half H of a 512-thread CTA (threads 256 H .. 256 H + 255)
// solving a zone of its own: its barrier is the named barrier 1 + H, its
// reductions run over its 8 warps through its own red / redd slices (32
// floats, 8 doubles; each slot is rewritten only after another of the
// half's barriers).  Sums are identical in every thread of the half.
template <int H>
struct HalfGroup {
    static constexpr int SIZE = 256;
    __device__ static void sum3h(float a, float b, float c, float *scr, float &sa, float &sb, float &sc) {
        group_halve3<8>(a, b, c, scr, (threadIdx.x >> 5) & 7, [] { sync(); }, sa, sb, sc);
    }
    __device__ static int rank() { return threadIdx.x - 256 * H; }
    __device__ static int size() { return 256; }
    __device__ static void sync() { asm volatile("bar.sync %0, 256;" ::"n"(1 + H) : "memory"); }
    __device__ static void sum3(float a, float b, float c, float *red, float &sa, float &sb,
                                float &sc) {
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
            c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) & 7;
        if (lane == 0) {
            red[3 * w] = a;
            red[3 * w + 1] = b;
            red[3 * w + 2] = c;
        }
        sync();
        float x = lane < 8 ? red[3 * lane] : 0.f;
        float y = lane < 8 ? red[3 * lane + 1] : 0.f;
        float q = lane < 8 ? red[3 * lane + 2] : 0.f;
#pragma unroll
        for (int o = 4; o; o >>= 1) {
            x += __shfl_xor_sync(0xffffffffu, x, o);
            y += __shfl_xor_sync(0xffffffffu, y, o);
            q += __shfl_xor_sync(0xffffffffu, q, o);
        }
        sa = __shfl_sync(0xffffffffu, x, 0);
        sb = __shfl_sync(0xffffffffu, y, 0);
        sc = __shfl_sync(0xffffffffu, q, 0);
    }
    __device__ static double sum(double x, double *redd) {
#pragma unroll
        for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        x = __shfl_sync(0xffffffffu, x, 0);
        if ((threadIdx.x & 31) == 0) redd[(threadIdx.x >> 5) & 7] = x;
        sync();
        double s = redd[threadIdx.x & 7];
#pragma unroll
        for (int o = 4; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        sync();
        return s;
    }
};

// z = P^-1 r for the rows of one group (block-Jacobi over rows sharing x0)
template <class V>
__device__ __forceinline__ void cg_precond_group(const V &v, int g) {
    const int a = v.gst[g] - v.goff, b = v.gst[g + 1] - v.goff;
    float rr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) rr[q] = a + q < b ? v.r[a + q] : 0.f;
    for (int t = a; t < b; ++t) {
        float4 m = v.pinv[t];
        v.z[t] = m.x * rr[0] + m.y * rr[1] + m.z * rr[2] + m.w * rr[3];
    }
}

// z = P^-1 r with P the blocks of rows sharing x0 or a face: one place of
// the block order per thread, its row of the block's inverse (four float4
// loads) against the block's residuals, summed in column order
constexpr int BLOCK_MAX = 16;

__host__ __device__ constexpr int tri(int i) { return i * (i + 1) / 2; }

template <class Gp, class V>
__device__ __forceinline__ void cg_precond_blocks(const V &v, int k) {
    for (int q = Gp::rank(); q < k; q += Gp::size()) {
        const int info = v.binfo[q];
        const int r0 = info >> 5, m = info & 31;
        const float4 *row = (const float4 *)(v.binv + 16 * (size_t)q);
        float c[BLOCK_MAX];
#pragma unroll
        for (int t = 0; t < BLOCK_MAX / 4; ++t) {
            const float4 x = t * 4 < m ? row[t] : make_float4(0.f, 0.f, 0.f, 0.f);
            c[4 * t] = x.x;
            c[4 * t + 1] = x.y;
            c[4 * t + 2] = x.z;
            c[4 * t + 3] = x.w;
        }
        float acc = 0.f;
#pragma unroll
        for (int t = 0; t < BLOCK_MAX; ++t)
            if (t < m) acc += c[t] * v.r[v.bperm[r0 + t]];
        v.z[v.bperm[q]] = acc;
    }
}

// A vertex's list is summed by one thread, the list of a hub (more than HUB_LIST
// entries) by its warp: a response around a hub of 300 rows 460 -> 365 us, of
// 1,300 2,510 -> 1,420 (with the early rejection of its matrix, solve_zone_rows).
// A warp sums its hubs one after another, so shorter lists stay with the
// threads, which sum 32 at a time (with 32 here a repair step of 1,024 pairs of
// spheres, whose coarse ones have lists of 40 to 60, took 2,048 us for 1,938).
constexpr int HUB_LIST = 128;

// whether one of this warp's vertices is a hub
template <class Gp, class V>
__device__ __forceinline__ bool cg_hubs(const V &v, int U) {
    bool hub = false;
    for (int j = Gp::rank(); j < U; j += Gp::size()) hub = hub || (int)v.seg[j + 1] - (int)v.seg[j] > HUB_LIST;
    return __any_sync(0xffffffffu, hub);
}

template <class Gp, class V>
__device__ __forceinline__ void cg_matvec_vertex(const V &v, int U, bool hubs) {
    const float third = 1.0f / 3.0f;
    // u of vertex j, its list's entries from, from + step, ... below e1 added up
    auto sum = [&](int from, int e1, int step, float &a0, float &a1, float &a2) {
        for (int e = from; e < e1; e += step) {
            int c = (int)v.cval[e] - v.coff;
            int s = c >> 2;
            float ps = ((c & 3) ? -third : 1.0f) * v.z[s];
            float3 n = v.nrm(s);
            a0 += ps * n.x;
            a1 += ps * n.y;
            a2 += ps * n.z;
        }
    };
    for (int j = Gp::rank(); j < U; j += Gp::size()) {
        float a0 = 0.f, a1 = 0.f, a2 = 0.f;
        const int e0 = (int)v.seg[j] - v.eoff, e1 = (int)v.seg[j + 1] - v.eoff;
        if (hubs && e1 - e0 > HUB_LIST) continue;
        sum(e0, e1, 1, a0, a1, a2);
        float w = v.winv[j];
        v.u[j] = make_float4(w * a0, w * a1, w * a2, 0.f);
    }
    if (!hubs) return;
    const int lane = threadIdx.x & 31;
    for (int j0 = Gp::rank() - lane; j0 < U; j0 += Gp::size()) {
        const int j = j0 + lane;
        const int e0 = j < U ? (int)v.seg[j] - v.eoff : 0, e1 = j < U ? (int)v.seg[j + 1] - v.eoff : 0;
        for (unsigned m = __ballot_sync(0xffffffffu, e1 - e0 > HUB_LIST); m; m &= m - 1u) {
            const int o = __ffs(m) - 1, h0 = __shfl_sync(0xffffffffu, e0, o), h1 = __shfl_sync(0xffffffffu, e1, o);
            float a0 = 0.f, a1 = 0.f, a2 = 0.f;
            sum(h0 + lane, h1, 32, a0, a1, a2);
#pragma unroll
            for (int q = 16; q; q >>= 1) {
                a0 += __shfl_xor_sync(0xffffffffu, a0, q);
                a1 += __shfl_xor_sync(0xffffffffu, a1, q);
                a2 += __shfl_xor_sync(0xffffffffu, a2, q);
            }
            if (lane == o) {
                float w = v.winv[j];
                v.u[j] = make_float4(w * a0, w * a1, w * a2, 0.f);
            }
        }
    }
}

template <class V>
__device__ __forceinline__ float cg_matvec_stencil(const V &v, int s) {
    const float third = 1.0f / 3.0f;
    int4 g = as_int4(v.vidx[s]);
    g.x -= v.voff; g.y -= v.voff; g.z -= v.voff; g.w -= v.voff;
    float3 n = v.nrm(s);
    float4 u0 = v.u[g.x], u1 = v.u[g.y], u2 = v.u[g.z], u3 = v.u[g.w];
    float d0 = u0.x - (u1.x + u2.x + u3.x) * third;
    float d1 = u0.y - (u1.y + u2.y + u3.y) * third;
    float d2 = u0.z - (u1.z + u2.z + u3.z) * third;
    return n.x * d0 + n.y * d1 + n.z * d2;
}

// returns the iteration count; x holds the solution of A x = r0
// Preconditioned CG in the Chronopoulos-Gear form (one fused reduction per
// iteration): u = P^-1 r, w = A u, s = A p by recurrence.  P is the
// block-Jacobi preconditioner over the groups.  Stops when |r| <= tol |r0|.
// Returns the iteration count; x holds the solution of A x = r0.
template <class Gp, class V>
__device__ __forceinline__ int cg_cg_loop(const V &v, int k, int U, int maxit, float tol,
                                          float *red) {
    const int tid = Gp::rank(), nt = Gp::size();
    const bool hubs = cg_hubs<Gp>(v, U);
    if (v.bperm) {
        cg_precond_blocks<Gp>(v, k);
    } else {
        for (int g = tid; g < v.G; g += nt) cg_precond_group(v, g);
    }
    Gp::sync();
    cg_matvec_vertex<Gp>(v, U, hubs);
    Gp::sync();
    float ga = 0.f, de = 0.f, rh = 0.f;
    for (int s = tid; s < k; s += nt) {
        float ws = cg_matvec_stencil(v, s);
        float rs = v.r[s], zs = v.z[s];
        v.w[s] = ws;
        ga += rs * zs;
        de += ws * zs;
        rh += rs * rs;
    }
    float gamma, delta, rho;
    Gp::sum3(ga, de, rh, red, gamma, delta, rho);
    const float stop = tol * tol * rho;
    float alpha = gamma / delta, beta = 0.f;
    int it = 0;
    while (it < maxit && rho > stop && rho > 0.f && alpha > 0.f && isfinite(alpha)) {
        if (v.bperm) {
            // the blocks span rows of other threads: the update, a barrier,
            // then the blocks
            for (int s = tid; s < k; s += nt) {
                const float ps = v.z[s] + beta * v.p[s];
                const float ss = v.w[s] + beta * v.sv[s];
                v.p[s] = ps;
                v.sv[s] = ss;
                v.x[s] += alpha * ps;
                v.r[s] -= alpha * ss;
            }
            Gp::sync();
            cg_precond_blocks<Gp>(v, k);
        } else {
            for (int g = tid; g < v.G; g += nt) {
                const int a = v.gst[g] - v.goff, b = v.gst[g + 1] - v.goff;
                for (int s = a; s < b; ++s) {
                    float ps = v.z[s] + beta * v.p[s];
                    float ss = v.w[s] + beta * v.sv[s];
                    v.p[s] = ps;
                    v.sv[s] = ss;
                    v.x[s] += alpha * ps;
                    v.r[s] -= alpha * ss;
                }
                cg_precond_group(v, g);
            }
        }
        Gp::sync();
        cg_matvec_vertex<Gp>(v, U, hubs);
        Gp::sync();
        ga = 0.f;
        de = 0.f;
        rh = 0.f;
        for (int s = tid; s < k; s += nt) {
            float ws = cg_matvec_stencil(v, s);
            float rs = v.r[s], zs = v.z[s];
            v.w[s] = ws;
            ga += rs * zs;
            de += ws * zs;
            rh += rs * rs;
        }
        float gn, dn, rn;
        Gp::sum3(ga, de, rh, red, gn, dn, rn);
        beta = gn / gamma;
        alpha = gn / (dn - beta * gn / alpha);
        gamma = gn;
        rho = rn;
        ++it;
    }
    return it;
}

// ---------------------------------------------------------------------------
// impact zones (Sec. 4: constraints with overlapping stencils form one
// zone, and each zone is one linear system).  Lock-free union-find over the
// stencils that share a vertex: a root is only ever hooked under a smaller
// root (atomicCAS), so each zone ends with its smallest stencil index as
// root; path halving only rewrites non-root entries with an ancestor.
// ---------------------------------------------------------------------------

__device__ __forceinline__ int uf_find(int *parent, int x) {
    while (true) {
        int p = __ldcg(parent + x);
        if (p == x) return x;
        int gp = __ldcg(parent + p);
        if (gp != p) parent[x] = gp;
        x = p;
    }
}

// Inputs of up to UF_SMALL stencils: one CTA runs the whole union-find in
// shared memory (the same hooking rule as below, so the same labels) and
// writes the zone keys; the global-memory kernels then return at once.
constexpr int UF_SMALL = 12288;  // 48 KB of parents

__device__ __forceinline__ int uf_find_s(volatile int *par, int x) {
    while (true) {
        const int p = par[x];
        if (p == x) return x;
        const int gp = par[p];
        if (gp != p) par[x] = gp;
        x = p;
    }
}

__global__ void __launch_bounds__(1024) k_uf_small(const int *d_k, const int *d_U, const int *seg,
                                                   const int *cval, unsigned *zlab, int *zsrc,
                                                   uint32_t *status) {
    HFCR_PDL_WAIT();
    __shared__ int par[UF_SMALL];
    const int k = *d_k;
    if (k > UF_SMALL) return;
    for (int i = threadIdx.x; i < k; i += blockDim.x) par[i] = i;
    __syncthreads();
    const int U = *d_U;
    for (int j = threadIdx.x; j < U; j += blockDim.x) {
        const int e0 = seg[j], e1 = seg[j + 1];
        const int s0 = cval[e0] >> 2;
        for (int e = e0 + 1; e < e1; ++e) {
            int a = s0, b = cval[e] >> 2;
            int guard = 0;
            while (true) {
                a = uf_find_s(par, a);
                b = uf_find_s(par, b);
                if (a == b) break;
                if (a < b) { int t = a; a = b; b = t; }
                const int old = atomicCAS(par + a, a, b);
                if (old == a) break;
                a = old;
                if (++guard > (1 << 24)) { atomicOr(status, ST_TIMEOUT); break; }
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < k; i += blockDim.x) {
        zlab[i] = (unsigned)uf_find_s(par, i);
        zsrc[i] = i;
    }
}

__global__ void k_uf_init(const int *d_k, int *parent) {
    HFCR_PDL_WAIT();
    const int k = *d_k;
    if (k <= UF_SMALL) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < k; i += gridDim.x * blockDim.x)
        parent[i] = i;
}

// unions the stencils of every touched vertex (CSR by vertex)
__global__ void k_uf_union(const int *d_k, const int *d_U, const int *seg, const int *cval,
                           int *parent, uint32_t *status) {
    HFCR_PDL_WAIT();
    if (*d_k <= UF_SMALL) return;
    const int U = *d_U;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < U; j += gridDim.x * blockDim.x) {
        const int e0 = seg[j], e1 = seg[j + 1];
        const int s0 = cval[e0] >> 2;
        for (int e = e0 + 1; e < e1; ++e) {
            int a = s0, b = cval[e] >> 2;
            // every failed exchange means another thread hooked that root:
            // the count of roots falls, so the loop ends; the bound is a guard
            int guard = 0;
            while (true) {
                a = uf_find(parent, a);
                b = uf_find(parent, b);
                if (a == b) break;
                if (a < b) { int t = a; a = b; b = t; }
                int old = atomicCAS(parent + a, a, b);
                if (old == a) break;
                a = old;
                if (++guard > (1 << 24)) { atomicOr(status, ST_TIMEOUT); break; }
            }
        }
    }
}

// zone label of every stencil (its root = the smallest stencil of its zone)
__global__ void k_zone_keys(const int *d_k, int *parent, unsigned *zlab, int *zsrc) {
    HFCR_PDL_WAIT();
    const int k = *d_k;
    if (k <= UF_SMALL) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < k; i += gridDim.x * blockDim.x) {
        zlab[i] = (unsigned)uf_find(parent, i);
        zsrc[i] = i;
    }
}

__global__ void k_zone_flags(const int *d_k, const unsigned *zlab, unsigned *flags) {
    HFCR_PDL_WAIT();
    const int k = *d_k;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < k; t += gridDim.x * blockDim.x)
        flags[t] = (t == 0 || zlab[t] != zlab[t - 1]) ? 1u : 0u;
}

// regroups the rows zone by zone (zones in the order of their smallest
// stencil, stencils ascending inside a zone: the label sort is stable)
__global__ void k_zone_gather(const int *d_k, const unsigned *zlab, const int *zsrc,
                              const unsigned *excl, const int4 *ids_raw,
                              const double4_32a *n64_raw, const float4 *n32_raw,
                              const double *b_raw, int4 *ids, double4_32a *n64, float4 *n32,
                              double *b, int *szone, int *zs, int *pos_of) {
    HFCR_PDL_WAIT();
    const int k = *d_k;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < k; t += gridDim.x * blockDim.x) {
        int src = zsrc[t];
        unsigned f = (t == 0 || zlab[t] != zlab[t - 1]) ? 1u : 0u;
        int z = (int)(excl[t] + f) - 1;
        szone[t] = z;
        pos_of[src] = t;
        if (f) zs[z] = t;
        if (t == k - 1) zs[z + 1] = k;
        ids[t] = ids_raw[src];
        n64[t] = n64_raw[src];
        n32[t] = n32_raw[src];
        b[t] = b_raw[src];
    }
}

// Zone-ordered CSR: the vertex-ordered entries (s * 4 + role) are re-sorted
// stably by the zone of their stencil, so vertices come out grouped by zone
// (vertex order kept inside a zone) and entries renumbered to zone order.
__global__ void k_csr2_entries(const int *cv1, const int *pos_of, const int *szone,
                               const int *d_k, int cap, unsigned *key, int *val) {
    HFCR_PDL_WAIT();
    int k = min(*d_k, cap);
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 4 * k) return;
    int e = cv1[i];
    int t = pos_of[e >> 2];
    key[i] = (unsigned)szone[t];
    val[i] = 4 * t + (e & 3);
}

__global__ void k_csr2_flags(const int *val, const int4 *ids, const int *d_k, int cap,
                             unsigned *flag) {
    HFCR_PDL_WAIT();
    int n = 4 * min(*d_k, cap);
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        flag[i] = (i == 0 || ((const int *)ids)[val[i]] != ((const int *)ids)[val[i - 1]]) ? 1u : 0u;
}

__global__ void k_csr2_build(const unsigned *zkey, const int *val, const unsigned *excl,
                             const int4 *ids, const int *d_k, int cap, int nA, const float *wA,
                             const float *wB, int4 *vidx, int *seg, int *gvert, float *winv,
                             int *zv, const int *d_nz) {
    HFCR_PDL_WAIT();
    int n = 4 * min(*d_k, cap);
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int g = ((const int *)ids)[val[i]];
    unsigned f = (i == 0 || g != ((const int *)ids)[val[i - 1]]) ? 1u : 0u;
    int j = (int)(excl[i] + f) - 1;
    ((int *)vidx)[val[i]] = j;
    if (f) {
        seg[j] = i;
        gvert[j] = g;
        const float *w = g < nA ? wA : wB;
        int lv = g < nA ? g : g - nA;
        winv[j] = w ? w[lv] : 1.0f;
        if (i == 0 || zkey[i] != zkey[i - 1]) zv[zkey[i]] = j;
    }
    if (i == n - 1) {
        seg[j + 1] = n;
        zv[*d_nz] = j + 1;
    }
}

// ---------------------------------------------------------------------------
// block-Jacobi preconditioner: rows whose stencils share x0 (an edge
// endpoint crossing several faces) are nearly dependent; they are
// contiguous inside a zone (stencils are sorted by (dir, x0, face)) and are
// grouped, at most GMAX rows per group.  Each group's block of A is inverted
// once per solve.
// ---------------------------------------------------------------------------
constexpr int GMAX = 4;

__device__ __forceinline__ bool group_start(const int4 *ids, const int *szone, const int *zs,
                                            int t) {
    const int zs0 = zs[szone[t]], x0 = ids[t].x;
    int rs = t;
    while (rs > zs0 && ids[rs - 1].x == x0) --rs;
    return ((t - rs) % GMAX) == 0;
}

__global__ void k_group_flags(const int *d_k, const int4 *ids, const int *szone, const int *zs,
                              unsigned *flags) {
    HFCR_PDL_WAIT();
    const int k = *d_k;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < k; t += gridDim.x * blockDim.x)
        flags[t] = group_start(ids, szone, zs, t) ? 1u : 0u;
}

__global__ void k_group_build(const int *d_k, const int4 *ids, const int *szone, const int *zs,
                              const unsigned *excl, const int *d_nz, int *gst, int *zg) {
    HFCR_PDL_WAIT();
    const int k = *d_k;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < k; t += gridDim.x * blockDim.x) {
        const bool st = group_start(ids, szone, zs, t);
        const int g = (int)excl[t];
        if (st) {
            gst[g] = t;
            const int z = szone[t];
            if (zs[z] == t) zg[z] = g;
        }
        if (t == k - 1) {
            const int ng = g + (st ? 1 : 0);
            gst[ng] = k;
            zg[*d_nz] = ng;
        }
    }
}

// inverse mass of global vertex g (1 where the mesh gives none)
__device__ __forceinline__ double inv_mass_of(int g, int nA, const float *wA, const float *wB) {
    const float *w = g < nA ? wA : wB;
    return w ? (double)w[g < nA ? g : g - nA] : 1.0;
}

// inverse of each group's block of A = J M^-1 J^T (float64, stored float32):
// A_ab = (n_a . n_b) (w(x0) + 1/9 sum of w over the face vertices shared by
// a and b); ids are the global vertex ids (x0, face) of the zone-ordered rows
__device__ __forceinline__ void store_inv_row(float4 *p, const double *row) {
    *p = make_float4((float)row[0], (float)row[1], (float)row[2], (float)row[3]);
}
__device__ __forceinline__ void store_inv_row(double4_32a *p, const double *row) {
    *p = make_double4_32a(row[0], row[1], row[2], row[3]);
}

// w / 9, without the division where there are no masses
__device__ __forceinline__ double ninth(double w) { return w == 1.0 ? 1.0 / 9.0 : w / 9.0; }

// Groups first .. n - 1, shared out over nw warps (this is warp wi), eight per
// warp: the four lanes of a quad hold the block's rows and run Gauss-Jordan with
// partial pivoting in registers, exchanging rows by shuffles.  A (near-)
// singular block falls back to the inverse of its diagonal.  Called by whole
// warps.  Bound by the latency of the loads and of float64 arithmetic: one
// thread per group with the block in local memory took 33 us (1,000 to 2,000
// groups), a quad 14 us.  Where few warps have many groups each (the
// cooperative setup just above what one CTA sets up), 32 groups of one row are
// taken at once, a lane each, with the bits of the quads: a response to 4,097
// stencils 528 -> 483 us.  R: float4 rows for the mixed solver, double4_32a rows
// for the float64 one; perm: row t is row perm[t] of ids and n64.
template <class G, typename R>
__device__ __forceinline__ void group_inverses(int first, int wi, int nw, int n, const int *gst, const int4 *ids,
                                               const double4_32a *n64, int nA, const float *wA,
                                               const float *wB, R *pinv, const int *perm = nullptr) {
    static_assert(GMAX == 4, "a quad holds one block");
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = threadIdx.x & 31, a = lane & 3, q0 = lane & ~3;
    const int per = n - first > 24 * nw ? 32 : 8;
    for (int g8 = first + per * wi; g8 < n;) {
        if (per == 32 && (g8 - first) % 32 == 0) {
            const int g = g8 + lane;
            const int a0 = g < n ? G::ld(gst + g) : 0, m = g < n ? G::ld(gst + g + 1) - a0 : 0;
            if (!__any_sync(ALL, m > 1)) {
                if (m == 1) {
                    const int t = perm ? G::ld(perm + a0) : a0;
                    const int4 v = G::ld(ids + t);
                    const double4_32a nv = ld_n64<G>(n64 + t);
                    const double w0 = inv_mass_of(v.x, nA, wA, wB), w1 = inv_mass_of(v.y, nA, wA, wB),
                                 w2 = inv_mass_of(v.z, nA, wA, wB), w3 = inv_mass_of(v.w, nA, wA, wB);
                    const int f[3] = {v.y, v.z, v.w};
                    const double d[3] = {ninth(w1), ninth(w2), ninth(w3)};
                    double w = w0;
#pragma unroll
                    for (int p = 0; p < 3; ++p)
#pragma unroll
                        for (int q = 0; q < 3; ++q)
                            if (f[p] == f[q]) w += d[p];
                    const double A = (nv.x * nv.x + nv.y * nv.y + nv.z * nv.z) * w;
                    double row[GMAX] = {0.0, 0.0, 0.0, 0.0};
                    if (fabs(A) > 1e-12 * fabs(A)) {
                        row[0] = 1.0 / A;
                    } else {
                        const double x = w0 + (w1 + w2 + w3) / 9.0;
                        row[0] = x > 0.0 ? 1.0 / x : 0.0;
                    }
                    store_inv_row(pinv + a0, row);
                }
                g8 += 32 * nw;
                continue;
            }
        }
        const int g = g8 + (lane >> 2);
        // eight groups further, behind the last of this warp's 32 (or 8) its next ones
        g8 += (g8 - first) % per == per - 8 ? per * nw - per + 8 : 8;
        const int a0 = g < n ? G::ld(gst + g) : 0, m = g < n ? G::ld(gst + g + 1) - a0 : 0;
        const int mmax = (int)__reduce_max_sync(ALL, (unsigned)m);
        int4 v = make_int4(0, 0, 0, 0);
        double4_32a nv = make_double4_32a(0.0, 0.0, 0.0, 0.0);
        double w0 = 0.0, w1 = 0.0, w2 = 0.0, w3 = 0.0;  // inverse masses of x0 and the face
        if (a < m) {
            const int t = perm ? G::ld(perm + a0 + a) : a0 + a;
            v = G::ld(ids + t);
            nv = ld_n64<G>(n64 + t);
            w0 = inv_mass_of(v.x, nA, wA, wB);
            w1 = inv_mass_of(v.y, nA, wA, wB);
            w2 = inv_mass_of(v.z, nA, wA, wB);
            w3 = inv_mass_of(v.w, nA, wA, wB);
        }
        const double d1 = ninth(w1), d2 = ninth(w2), d3 = ninth(w3);
        double A[2 * GMAX], diag = 0.0;
#pragma unroll
        for (int b = 0; b < GMAX; ++b) {
            A[b] = 0.0;
            A[GMAX + b] = 0.0;
            if (b >= mmax) continue;
            const int fb[3] = {__shfl_sync(ALL, v.y, q0 + b), __shfl_sync(ALL, v.z, q0 + b),
                               __shfl_sync(ALL, v.w, q0 + b)};
            const double bx = __shfl_sync(ALL, nv.x, q0 + b), by = __shfl_sync(ALL, nv.y, q0 + b),
                         bz = __shfl_sync(ALL, nv.z, q0 + b);
            if (a >= m || b >= m) continue;
            double w = w0;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (v.y == fb[q]) w += d1;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (v.z == fb[q]) w += d2;
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (v.w == fb[q]) w += d3;
            A[b] = (nv.x * bx + nv.y * by + nv.z * bz) * w;
            A[GMAX + b] = a == b ? 1.0 : 0.0;
            if (a == b) diag = fabs(A[b]);
        }
        double dmax = fmax(diag, __shfl_xor_sync(ALL, diag, 1));
        dmax = fmax(dmax, __shfl_xor_sync(ALL, dmax, 2));
        bool ok = true;
#pragma unroll
        for (int c = 0; c < GMAX; ++c) {
            if (c >= mmax) break;
            const double mag = fabs(A[c]);
            int piv = c;
            double best = __shfl_sync(ALL, mag, q0 + c);
#pragma unroll
            for (int r = c + 1; r < GMAX; ++r) {
                const double o = __shfl_sync(ALL, mag, q0 + r);
                if (r < m && o > best) {
                    piv = r;
                    best = o;
                }
            }
            if (c < m && !(best > 1e-12 * dmax)) ok = false;
            const bool act = c < m && ok;
            if (__any_sync(ALL, act && piv != c)) {
                const int from = q0 + (act && a == c ? piv : act && a == piv ? c : a);
#pragma unroll
                for (int q = 0; q < 2 * GMAX; ++q) A[q] = __shfl_sync(ALL, A[q], from);
            }
            if (act && a == c) {
                const double inv = 1.0 / A[c];
#pragma unroll
                for (int q = 0; q < 2 * GMAX; ++q) A[q] *= inv;
            }
            if (mmax == 1) break;  // no other rows
            const double f = A[c];
#pragma unroll
            for (int q = 0; q < 2 * GMAX; ++q) {
                const double p = __shfl_sync(ALL, A[q], q0 + c);
                if (act && a != c) A[q] -= f * p;
            }
        }
        if (a < m) {
            double row[GMAX];
#pragma unroll
            for (int b = 0; b < GMAX; ++b) row[b] = A[GMAX + b];
            if (!ok) {
                const double w = w0 + (w1 + w2 + w3) / 9.0, x = w > 0.0 ? 1.0 / w : 0.0;
#pragma unroll
                for (int b = 0; b < GMAX; ++b) row[b] = a == b ? x : 0.0;
            }
            store_inv_row(pinv + a0 + a, row);
        }
    }
}

__global__ void k_group_inverse(const int *d_ng, const int *gst, const int4 *ids,
                                const double4_32a *n64, int nA, const float *wA, const float *wB,
                                float4 *pinv) {
    HFCR_PDL_WAIT();
    const int nw = blockDim.x >> 5;
    group_inverses<PlainLd>(0, (int)(blockIdx.x * nw + (threadIdx.x >> 5)), (int)gridDim.x * nw, *d_ng, gst,
                            ids, n64, nA, wA, wB, pinv);
}

// float64 residual r = b - J M^-1 J^T lam of one zone (the float64 normals;
// Eq. 7), written to v.r in float32 as the next right-hand side.  The
// vertex half goes through u64 (global scratch, this zone's rows only).
// Returns |r|^2, identical in every thread.
template <class Gp, class V>
__device__ __forceinline__ double zone_residual(const V &v, int k, int U, int s0, int j0,
                                                const double4_32a *n64, const double *b64,
                                                const double *lam, double *u64, double *redd) {
    const int tid = Gp::rank(), nt = Gp::size();
    const double third = 1.0 / 3.0;
    for (int j = tid; j < U; j += nt) {
        double a0 = 0.0, a1 = 0.0, a2 = 0.0;
        const int e1 = (int)v.seg[j + 1] - v.eoff;
        for (int e = (int)v.seg[j] - v.eoff; e < e1; ++e) {
            const int c = (int)v.cval[e] - v.coff;
            const int sl = c >> 2;
            const double ps = ((c & 3) ? -third : 1.0) * lam[s0 + sl];
            const double4_32a n = n64[s0 + sl];
            a0 += ps * n.x;
            a1 += ps * n.y;
            a2 += ps * n.z;
        }
        const double w = (double)v.winv[j];
        double *u = u64 + 3 * (size_t)(j0 + j);
        u[0] = w * a0;
        u[1] = w * a1;
        u[2] = w * a2;
    }
    Gp::sync();
    double rr = 0.0;
    for (int t = tid; t < k; t += nt) {
        const int4 g = as_int4(v.vidx[t]);
        const double *ux = u64 + 3 * (size_t)(j0 + g.x - v.voff);
        const double *ua = u64 + 3 * (size_t)(j0 + g.y - v.voff);
        const double *ub = u64 + 3 * (size_t)(j0 + g.z - v.voff);
        const double *uc = u64 + 3 * (size_t)(j0 + g.w - v.voff);
        const double4_32a n = n64[s0 + t];
        const double d0 = ux[0] - (ua[0] + ub[0] + uc[0]) * third;
        const double d1 = ux[1] - (ua[1] + ub[1] + uc[1]) * third;
        const double d2 = ux[2] - (ua[2] + ub[2] + uc[2]) * third;
        const double r = b64[s0 + t] - (n.x * d0 + n.y * d1 + n.z * d2);
        v.r[t] = (float)r;
        rr += r * r;
    }
    return Gp::sum(rr, redd);
}

// Arguments of the zone solvers (device pointers of the zone-ordered system).
struct ZoneArgs {
    const int *zs, *zv, *zg;       // zone starts of rows, touched vertices, groups
    const int *seg, *cval;         // vertex CSR (zone-contiguous)
    const float *winv;
    const float4 *n32, *pinv;
    const double4_32a *n64;
    const int4 *vidx;
    const int *gst;
    const double *b64;
    double *lam, *u64, *zres, *zbb;
    int maxit, max_refine;
    double tol, rel_tol;
    int *ctl;
    unsigned *ticket;  // [2] zone counters of the pair launch (zero before a solve)
    // float64 per-zone solve: rows' global vertex ids, inverse masses, and the
    // float64 inverse blocks it computes
    const int4 *ids;
    int nA;
    const float *wA, *wB;
    double4_32a *pinv64;  // [cap_k]
    float *binv;          // [16 cap_k] rows of the large zones' block inverses (mixed solver)
    int block_switch;     // iterations of a large zone's run before its blocks (-1: never)
};

// |b_zone|^2 with lam = 0 for the zone's rows
template <class Gp>
__device__ __forceinline__ double zone_start(const ZoneArgs &a, int s0, int k, double *redd) {
    double bb = 0.0;
    for (int t = Gp::rank(); t < k; t += Gp::size()) {
        const double bv = a.b64[s0 + t];
        bb += bv * bv;
        a.lam[s0 + t] = 0.0;
    }
    return Gp::sum(bb, redd);
}

// shared memory a zone needs for the staged solve: per row the float32
// normal, the preconditioner row, six CG vectors, four 16-bit CSR entries
// and 16-bit vertex ids (72 B); per touched vertex u, the inverse mass and
// a 16-bit CSR offset (22 B); per group its first row; alignment slack
__device__ __forceinline__ long long zone_smem_need(int k, int U, int G) {
    return 72ll * k + 22ll * U + 4ll * G + 48;
}

struct ZoneResult {
    double rr;   // final |r|^2 of the zone
    int its;     // CG iterations
    int rounds;  // float32 runs
};

// exclusive prefix sums of a[0 .. n) in place over the whole group (each
// thread a contiguous run, warp and group scans of the runs' totals);
// returns the total.  ws: 32 ints of scratch.
template <class Gp>
__device__ __forceinline__ int group_scan_excl(int *a, int n, int *ws) {
    const int tid = Gp::rank(), nt = Gp::size();
    const int lane = tid & 31, w = tid >> 5, nw = nt >> 5;
    const int per = (n + nt - 1) / nt, lo = tid * per, hi = lo + per < n ? lo + per : n;
    int sum = 0;
    for (int i = lo; i < hi; ++i) sum += a[i];
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[w] = x;
    Gp::sync();
    if (w == 0) {
        int t = lane < nw ? ws[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) ws[lane] = t;
    }
    Gp::sync();
    int run = (w > 0 ? ws[w - 1] : 0) + x - sum;
    const int total = ws[nw - 1];
    for (int i = lo; i < hi; ++i) {
        const int t = a[i];
        a[i] = run;
        run += t;
    }
    Gp::sync();
    return total;
}

// one union of the shared-memory union-find: the larger root is hooked
// under the smaller (so every zone's blocks are the same whatever the
// order of the unions); a lost race retries, at most a bounded number of
// times (a skipped union leaves two blocks where one would do: still a
// valid block preconditioner)
__device__ __forceinline__ void uf_union_s(int *par, int a, int b) {
    volatile int *vp = par;
    for (int tries = 0; tries < 4096; ++tries) {
        a = uf_find_s(vp, a);
        b = uf_find_s(vp, b);
        if (a == b) return;
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        if (atomicCAS(par + b, b, a) == b) return;
    }
}

// The inverse of one block of m <= N rows (rows[0 .. m)), in float64 (a
// block of nearly dependent rows has a large condition number, and its
// float32 inverse can come out indefinite): the matrix from the float32
// normals (products exact in float64), factored L L^T (the diagonal kept as
// 1 / L_ii; a pivot below 1e-12 of its diagonal entry makes the block its
// diagonal), L^-1, then L^-T L^-1, symmetric by construction, rounded to
// float32; row i to out + 16 i.  N fixes the unrolled bounds (a block pays
// for the size class it falls in).
template <int N, class V>
__device__ __forceinline__ void block_inverse(const V &v, const uint16_t *rows, int m, float *out) {
    const double third = 1.0 / 3.0;
    double Lr[tri(N)];
    bool ok = true;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if (i >= m) continue;
        const int si = rows[i];
        const ushort4 gi = v.vidx[si];
        const float3 ni = v.nrm(si);
        const int vi[4] = {gi.x, gi.y, gi.z, gi.w};
#pragma unroll
        for (int j = 0; j <= i; ++j) {
            const int sj = rows[j];
            const ushort4 gj = v.vidx[sj];
            const float3 nj = v.nrm(sj);
            const int vj[4] = {gj.x, gj.y, gj.z, gj.w};
            double wsh = 0.0;
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (vi[p] == vj[q]) wsh += (p ? -third : 1.0) * (q ? -third : 1.0) * (double)v.winv[vi[p]];
            const double dot = (double)ni.x * nj.x + (double)ni.y * nj.y + (double)ni.z * nj.z;
            double a_ij = dot * wsh;
            const double a_ii = a_ij;
#pragma unroll
            for (int q = 0; q < j; ++q) a_ij -= Lr[tri(i) + q] * Lr[tri(j) + q];
            if (j < i) {
                Lr[tri(i) + j] = a_ij * Lr[tri(j) + j];
            } else if (ok && a_ij > 1e-12 * a_ii && isfinite(a_ij)) {
                Lr[tri(i) + i] = rsqrt(a_ij);
            } else {
                ok = false;
            }
        }
    }
    if (!ok) {
        // the block's diagonal alone
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if (i >= m) continue;
            const int si = rows[i];
            const ushort4 gi = v.vidx[si];
            const float3 ni = v.nrm(si);
            const int vi[4] = {gi.x, gi.y, gi.z, gi.w};
            double wsh = 0.0;
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (vi[p] == vi[q]) wsh += (p ? -third : 1.0) * (q ? -third : 1.0) * (double)v.winv[vi[p]];
            const double d = ((double)ni.x * ni.x + (double)ni.y * ni.y + (double)ni.z * ni.z) * wsh;
#pragma unroll
            for (int q = 0; q < i; ++q) Lr[tri(i) + q] = 0.0;
            Lr[tri(i) + i] = d > 0.0 && isfinite(d) ? rsqrt(d) : 1.0;
        }
    }
    double Li[tri(N)];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        if (j >= m) continue;
        Li[tri(j) + j] = Lr[tri(j) + j];
#pragma unroll
        for (int i = j + 1; i < N; ++i) {
            if (i >= m) continue;
            double t = 0.0;
#pragma unroll
            for (int q = j; q < i; ++q) t += Lr[tri(i) + q] * Li[tri(q) + j];
            Li[tri(i) + j] = -t * Lr[tri(i) + i];
        }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if (i >= m) continue;
#pragma unroll
        for (int j = 0; j <= i; ++j) {
            double t = 0.0;
#pragma unroll
            for (int q = i; q < N; ++q)
                if (q < m) t += Li[tri(q) + i] * Li[tri(q) + j];
            out[16 * i + j] = (float)t;
            out[16 * j + i] = (float)t;
        }
    }
}

// The inverse of one block of 4 < m <= BLOCK_MAX rows by one warp, in
// float64: lane j < 16 holds column j of the block's matrix, lane 16 + j
// column j of the identity; Gauss-Jordan elimination without pivoting (the
// matrix is symmetric positive definite), the pivot column broadcast by
// shuffles at each step, turns the right half into the inverse, which is
// written rounded to float32 and made symmetric pairwise; a pivot that is
// not positive makes the block its diagonal.  Called by every lane.
template <class V>
__device__ __forceinline__ void block_inverse_warp(const V &v, const uint16_t *rows, int m, float *out) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, j = lane & 15;
    const double third = 1.0 / 3.0;
    double c[BLOCK_MAX];
#pragma unroll
    for (int i = 0; i < BLOCK_MAX; ++i) c[i] = 0.0;
    if (lane < 16 && j < m) {
        const int sj = rows[j];
        const ushort4 gj = v.vidx[sj];
        const float3 nj = v.nrm(sj);
        const int vj[4] = {gj.x, gj.y, gj.z, gj.w};
#pragma unroll
        for (int i = 0; i < BLOCK_MAX; ++i) {
            if (i >= m) continue;
            const int si = rows[i];
            const ushort4 gi = v.vidx[si];
            const float3 ni = v.nrm(si);
            const int vi[4] = {gi.x, gi.y, gi.z, gi.w};
            double wsh = 0.0;
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (vi[p] == vj[q]) wsh += (p ? -third : 1.0) * (q ? -third : 1.0) * (double)v.winv[vi[p]];
            c[i] = ((double)ni.x * nj.x + (double)ni.y * nj.y + (double)ni.z * nj.z) * wsh;
        }
    } else if (lane >= 16 && j < m) {
#pragma unroll
        for (int i = 0; i < BLOCK_MAX; ++i)
            if (i == j) c[i] = 1.0;
    }
    double dj = 0.0;  // the block's diagonal entry of lane j (< 16), for the fallback
#pragma unroll
    for (int i = 0; i < BLOCK_MAX; ++i)
        if (i == j) dj = c[i];
    bool ok = true;
#pragma unroll
    for (int kk = 0; kk < BLOCK_MAX; ++kk) {
        if (kk >= m) break;
        const double piv = __shfl_sync(full, c[kk], kk);
        const double d0 = __shfl_sync(full, dj, kk);
        ok = ok && piv > 1e-12 * d0 && isfinite(piv);
        c[kk] *= 1.0 / piv;
#pragma unroll
        for (int i = 0; i < BLOCK_MAX; ++i) {
            if (i >= m || i == kk) continue;
            const double f = __shfl_sync(full, c[i], kk);
            c[i] -= f * c[kk];
        }
    }
    if (ok) {
        if (lane >= 16 && j < m) {
#pragma unroll
            for (int i = 0; i < BLOCK_MAX; ++i)
                if (i < m) out[16 * i + j] = (float)c[i];
        }
        __syncwarp();
        // (i, u) and (u, i) to their mean, the pair handled by lane i > u
        if (lane < m) {
            for (int u = 0; u < lane; ++u) {
                const float x = 0.5f * (out[16 * lane + u] + out[16 * u + lane]);
                out[16 * lane + u] = x;
                out[16 * u + lane] = x;
            }
        }
    } else if (lane < 16 && j < m) {
        for (int i = 0; i < m; ++i) out[16 * i + j] = i == j ? (dj > 0.0 && isfinite(dj) ? (float)(1.0 / dj) : 1.f) : 0.f;
    }
    __syncwarp();
}

// The preconditioner blocks of a staged large zone (Sec. 4's rows of one
// impact zone): rows joined when they share x0 or the face (their nearly
// parallel rows make the zone's system ill-conditioned, and a block that
// holds them all captures that); a component of at most BLOCK_MAX rows is
// one block, a larger one is cut into runs of whole x0 groups of at most
// BLOCK_MAX rows, in row order.  Rows are ordered by block
// (ascending within a block), and every block's matrix, entry (s, t) =
// (n_s . n_t) sum over the vertices v the two rows share of c_s(v) c_t(v)
// w(v) (c = 1 at x0, -1/3 at a face vertex), is factored L L^T in float32
// (a pivot that is not positive makes the block its diagonal) and inverted
// as L^-T L^-1, which is symmetric by construction; place q of the block
// order gets its row bperm[q], its block's start and size binfo[q] and its
// row of the inverse at binv + 16 q.  Called between rounds; scratch: the
// CG vectors p, sv, w, z and x (dead between rounds), bst (k + 1 ints) and
// 96 ints at ws.  Returns the block count.  Not inlined: its register
// needs (the unrolled factorisations) stay out of the CG loop's allocation.
template <class Gp>
__device__ __noinline__ int zone_blocks(const CgViewS &v, int k, int U, const int *gst, int G,
                                           uint16_t *bperm, int *binfo, int *bst, float *binv,
                                           int *ws) {
    const int tid = Gp::rank(), nt = Gp::size();
    int *par = (int *)v.p;   // [k] union-find parents, then each row's block key
    int *cnt = (int *)v.sv;  // [k] component sizes, then block numbers of the keys
    int *hist = (int *)v.w;  // [k + 1] rows per key (w and z are contiguous)
    for (int t = tid; t < k; t += nt) {
        par[t] = t;
        cnt[t] = 0;
    }
    for (int t = tid; t <= k; t += nt) hist[t] = 0;
    Gp::sync();
    // rows with the same x0 are neighbours in the zone's order (dir, x0, face)
    for (int t = 1 + tid; t < k; t += nt)
        if (v.vidx[t].x == v.vidx[t - 1].x) uf_union_s(par, t, t - 1);
    // rows with the same face both list its first vertex in role 1
    for (int j = tid; j < U; j += nt) {
        const int e0 = v.seg[j], e1 = v.seg[j + 1];
        for (int e = e0; e < e1; ++e) {
            const int c = v.cval[e];
            if ((c & 3) != 1) continue;
            const ushort4 gs = v.vidx[c >> 2];
            for (int f = e + 1; f < e1; ++f) {
                const int c2 = v.cval[f];
                if ((c2 & 3) != 1) continue;
                const ushort4 gt = v.vidx[c2 >> 2];
                if (gs.z == gt.z && gs.w == gt.w) uf_union_s(par, c >> 2, c2 >> 2);
            }
        }
    }
    Gp::sync();
    for (int t = tid; t < k; t += nt) par[t] = uf_find_s((volatile int *)par, t);
    Gp::sync();
    for (int t = tid; t < k; t += nt) atomicAdd(&cnt[par[t]], 1);
    int *keys = (int *)v.x;  // the block key of each row (x is dead between rounds)
    int *nbig = ws + 32, *big = ws + 33;
    if (tid == 0) *nbig = 0;
    Gp::sync();
    // the components of more than BLOCK_MAX rows (up to 63 of them)
    for (int t = tid; t < k; t += nt)
        if (par[t] == t && cnt[t] > BLOCK_MAX) {
            const int i = atomicAdd(nbig, 1);
            if (i < 63) big[i] = t;
        }
    // block key of a row: its component's root; in a larger component the
    // first row of its x0 group, unless that component is split below
    for (int g = tid; g < G; g += nt)
        for (int t = gst[g]; t < gst[g + 1]; ++t) {
            const int r = par[t];
            keys[t] = cnt[r] <= BLOCK_MAX ? r : gst[g];
        }
    Gp::sync();
    // a listed large component in runs of whole x0 groups, in row order, of
    // at most BLOCK_MAX rows (one thread a component; the key of a run is
    // its first row)
    const int nb_list = *nbig < 63 ? *nbig : 63;
    for (int c = tid; c < nb_list; c += nt) {
        const int r = big[c];
        int acc = 0, key = -1;
        for (int g = 0; g < G; ++g) {
            const int t0 = gst[g];
            if (par[t0] != r) continue;
            const int sz = gst[g + 1] - t0;
            if (key < 0 || acc + sz > BLOCK_MAX) {
                key = t0;
                acc = 0;
            }
            acc += sz;
            for (int t = t0; t < t0 + sz; ++t) keys[t] = key;
        }
    }
    Gp::sync();
    for (int t = tid; t < k; t += nt) atomicAdd(&hist[keys[t]], 1);
    Gp::sync();
    group_scan_excl<Gp>(hist, k + 1, ws);  // hist[key]: first place of the key's rows
    for (int q = tid; q < k; q += nt) cnt[q] = hist[q + 1] > hist[q] ? 1 : 0;
    Gp::sync();
    const int NB = group_scan_excl<Gp>(cnt, k, ws);
    for (int q = tid; q < k; q += nt)
        if (hist[q + 1] > hist[q]) bst[cnt[q]] = hist[q];
    if (tid == 0) bst[NB] = k;
    Gp::sync();
    for (int t = tid; t < k; t += nt) bperm[atomicAdd(&hist[keys[t]], 1)] = (uint16_t)t;
    Gp::sync();
    // one thread per block: its rows in ascending order, then the inverse of
    // a block of at most 4 rows; the larger ones are listed for the warps
    int *wlist = cnt;  // the block numbers are no longer needed
    int *nwl = ws + 32;
    if (tid == 0) *nwl = 0;
    Gp::sync();
    for (int b = tid; b < NB; b += nt) {
        const int r0 = bst[b], m = bst[b + 1] - r0;
        for (int i = 1; i < m; ++i) {
            const uint16_t x = bperm[r0 + i];
            int j = i - 1;
            while (j >= 0 && bperm[r0 + j] > x) {
                bperm[r0 + j + 1] = bperm[r0 + j];
                --j;
            }
            bperm[r0 + j + 1] = x;
        }
        for (int i = 0; i < m; ++i) binfo[r0 + i] = (r0 << 5) | m;
        if (m <= 4)
            block_inverse<4>(v, bperm + r0, m, binv + 16 * (size_t)r0);
        else
            wlist[atomicAdd(nwl, 1)] = b;  // for a warp below
    }
    Gp::sync();
    // the larger blocks, one warp each
    {
        const int nwarps = nt >> 5, w = tid >> 5, nl = *nwl;
        for (int i = w; i < nl; i += nwarps) {
            const int b = wlist[i], r0 = bst[b];
            block_inverse_warp(v, bperm + r0, bst[b + 1] - r0, binv + 16 * (size_t)r0);
        }
    }
    Gp::sync();
    return NB;
}

// Rounds of iterative refinement of zone z, everything the float32 CG
// touches staged in shared memory at base (zone_smem_need bytes); BLK: the
// large zones' preconditioner blocks (zone_blocks) instead of the groups.
// warm (BLK): lambda and res come from solve_zone_rows, whose run took
// block_switch iterations; the blocks take over from there.
template <class Gp, bool BLK = false>
__device__ __forceinline__ ZoneResult solve_zone_smem(const ZoneArgs &a, int z, char *base, double bb,
                                                      float *red, double *redd, const ZoneResult *warm = nullptr) {
    const int tid = Gp::rank(), nt = Gp::size();
    const int s0 = a.zs[z], k = a.zs[z + 1] - s0;
    const int j0 = a.zv[z], U = a.zv[z + 1] - j0;
    const int g0 = a.zg[z], G = a.zg[z + 1] - g0;
    const int e0 = a.seg[j0];
    const double target = a.rel_tol * a.rel_tol * bb;
    CgViewS v;
    // layout: n4 | pinv | u | r p x sv w z | winv | gst | vidx (16-bit) | seg (16-bit) | cval (16-bit)
    float4 *n4 = (float4 *)base;
    float4 *pinv = n4 + k;
    v.u = pinv + k;
    float *f = (float *)(v.u + U);
    v.r = f; v.p = f + k; v.x = f + 2 * k; v.sv = f + 3 * k; v.w = f + 4 * k; v.z = f + 5 * k;
    float *winv = f + 6 * k;
    int *gst = (int *)(winv + U);
    ushort4 *vidx = (ushort4 *)(((uintptr_t)(gst + G + 1) + 7) & ~(uintptr_t)7);
    uint16_t *seg = (uint16_t *)(vidx + k);
    uint16_t *cval = seg + U + 1;
    for (int t = tid; t < k; t += nt) {
        const int4 g = a.vidx[s0 + t];
        vidx[t] = make_ushort4((unsigned short)(g.x - j0), (unsigned short)(g.y - j0),
                               (unsigned short)(g.z - j0), (unsigned short)(g.w - j0));
        n4[t] = a.n32[s0 + t];
        pinv[t] = a.pinv[s0 + t];
        v.r[t] = (float)a.b64[s0 + t];
    }
    for (int g = tid; g <= G; g += nt) gst[g] = a.gst[g0 + g] - s0;
    v.pinv = pinv; v.gst = gst; v.G = G; v.goff = 0;
    for (int j = tid; j <= U; j += nt) seg[j] = (uint16_t)(a.seg[j0 + j] - e0);
    for (int j = tid; j < U; j += nt) winv[j] = a.winv[j0 + j];
    for (int e = tid; e < 4 * k; e += nt) cval[e] = (uint16_t)(a.cval[e0 + e] - 4 * s0);
    v.n4 = n4;
    v.vidx = vidx; v.seg = seg; v.cval = cval; v.winv = winv;
    v.voff = 0; v.coff = 0; v.eoff = 0;
    double rr = bb;
    int its = 0, rounds = 0, extra = 0;
    // BLK: a run stops after block_switch iterations; a zone that needs
    // more (an ill-conditioned one) keeps that run's correction and
    // continues on the blocks (that run is not counted)
    bool blocks_on = false;
    const bool may_switch = BLK && a.block_switch > 0 && a.block_switch < a.maxit;
    auto to_blocks = [&]() {
        // the block order, the places' blocks and the block starts in
        // the groups' inverse rows' slot (16 B a row: 2 + 4 + 4)
        uint16_t *bperm = (uint16_t *)pinv;
        int *binfo = (int *)(bperm + ((k + 7) & ~7));
        int *bst = binfo + k;
        float *binv = a.binv + 16 * (size_t)s0;
        zone_blocks<Gp>(v, k, U, gst, G, bperm, binfo, bst, binv, (int *)red);
        v.bperm = bperm;
        v.binfo = binfo;
        v.binv = binv;
        blocks_on = true;
        extra = 1;
    };
    if constexpr (BLK) {
        if (warm) {
            Gp::sync();
            rr = zone_residual<Gp>(v, k, U, s0, j0, a.n64, a.b64, a.lam, a.u64, redd);
            its = warm->its;
            rounds = warm->rounds;
            to_blocks();
        }
    }
    while (rr > target && rounds < a.max_refine + extra) {
        for (int t = tid; t < k; t += nt) {
            v.p[t] = 0.f;
            v.sv[t] = 0.f;
            v.x[t] = 0.f;
        }
        Gp::sync();
        const int cap_it = may_switch && !blocks_on ? a.block_switch : a.maxit;
        const int n_it = cg_cg_loop<Gp>(v, k, U, cap_it, (float)a.tol, red);
        its += n_it;
        for (int t = tid; t < k; t += nt) a.lam[s0 + t] += (double)v.x[t];
        Gp::sync();
        const double rr_prev = rr;
        rr = zone_residual<Gp>(v, k, U, s0, j0, a.n64, a.b64, a.lam, a.u64, redd);
        ++rounds;
        if (!(rr < rr_prev)) {
            // the run did not reduce the float64 residual (a stagnating or
            // failing float32 run): its correction is taken back, the zone
            // keeps the best lambda found
            for (int t = tid; t < k; t += nt) a.lam[s0 + t] -= (double)v.x[t];
            rr = rr_prev;
            Gp::sync();
            break;
        }
        if constexpr (BLK) {
            if (may_switch && !blocks_on && n_it >= cap_it && rr > target) to_blocks();
        }
    }
    ZoneResult res;
    res.rr = rr;
    res.its = its;
    res.rounds = rounds;
    return res;
}

// ---------------------------------------------------------------------------
// A zone solved by rows: the same rounds as solve_zone_smem (float32 PCG to
// inner_tol, float64 residual), with the zone's matrix A = J M^-1 J^T written
// out once.  Its rows are short (5 to 9 entries on average where cloth and
// bodies cross: few stencils share a vertex), so a product is one pass over a
// row's entries in the place of the vertex gather, a barrier and the four-
// vertex products.  Row t belongs to one thread (RPT rows each), which keeps
// the row's CG vectors, its inverse-block row and lambda in registers; only r
// (for the blocks) and z are exchanged through shared memory.  The entries,
// (value, column), lie in slices of 32 rows, as long as the slice's longest
// row and column by column, so that a warp reads them without conflicts.
// Bound by the latency of an iteration's three barriers and shared-memory
// passes: against a gather of u and four vertex products per row, a zone of
// 1,219 rows (74 iterations, 3 rounds) 440 -> 227 us, zones of 33 to 255 rows
// in pairs 185 -> 124 us, zones of up to 32 rows in a warp each 96 -> 45 us.
// On an ill-conditioned zone the rounds get weak: the entries are rounded, and
// so are the products of the other form.  Where a round reduces the float64
// residual by less than ROWS_WEAK and more than one such step is left, the zone
// is given to the float64 rescue at once if that is staged (rescue_fits): a zone
// of 354 rows left at 7e-6 went on for three rounds of 104 to 180 iterations
// before (its call 1.91 -> 1.27 ms).
// Returns 0 when done (res filled, lambda stored), 1 when the zone does not
// fit (rows, shared memory) and nothing was done, 2 when a run of a
// BLK zone took block_switch iterations: lambda holds the best so far, and the
// blocks are to take over.
// ---------------------------------------------------------------------------
constexpr double ROWS_WEAK = 30.0;

// the float64 rescue (zone64_staged): its threads with rows, the rows of each,
// its shared memory, and whether a zone fits `bytes` of it
constexpr int RESCUE_NT = 256, RESCUE_ROWS = 4;
constexpr int RESCUE_SMEM = 220 * 1024;
__device__ __forceinline__ bool rescue_fits(int k, int U, int bytes) {
    return k <= RESCUE_ROWS * RESCUE_NT && 98ll * k + 30ll * U + 64 <= bytes;
}

template <class Gp, int RPT, bool BLK>
__device__ __forceinline__ int solve_zone_rows(const ZoneArgs &a, int z, char *base, int bytes, double bb,
                                               float *red, double *redd, ZoneResult &res) {
    constexpr int NT = Gp::SIZE, NS = RPT * NT / 32;  // slices of 32 rows
    const int tid = Gp::rank(), lane = threadIdx.x & 31, wq = tid >> 5;
    const int s0 = a.zs[z], k = a.zs[z + 1] - s0;
    const int j0 = a.zv[z], U = a.zv[z + 1] - j0;
    const int g0 = a.zg[z], G = a.zg[z + 1] - g0;
    const int e0 = a.seg[j0];
    // layout: n4 (later r and z) | lambda and -lambda / 3 | vidx | winv | seg |
    // cval | groups | slices | matrix, u
    const long long fixed = 50ll * k + 6ll * U + 4ll * NS + 64;
    if (k > RPT * NT || fixed > bytes) return 1;
    float4 *n4 = (float4 *)base;
    float *rS = (float *)base, *zS = rS + k;
    double *lamS = (double *)(n4 + k);
    ushort4 *vidx = (ushort4 *)(lamS + 2 * k);
    float *winv = (float *)(vidx + k);
    uint16_t *seg = (uint16_t *)(winv + U);
    uint16_t *cval = seg + U + 1;
    uint16_t *grp = cval + 4 * k;
    int *sl = (int *)(((uintptr_t)(grp + k) + 3) & ~(uintptr_t)3);
    for (int t = tid; t < k; t += NT) {
        const int4 g = a.vidx[s0 + t];
        vidx[t] = make_ushort4((unsigned short)(g.x - j0), (unsigned short)(g.y - j0),
                               (unsigned short)(g.z - j0), (unsigned short)(g.w - j0));
        n4[t] = a.n32[s0 + t];
    }
    for (int g = tid; g < G; g += NT) {  // each row's block: first row and size
        const int b0 = a.gst[g0 + g] - s0, b1 = a.gst[g0 + g + 1] - s0;
        for (int t = b0; t < b1; ++t) grp[t] = (uint16_t)(b0 << 3 | (b1 - b0));
    }
    for (int j = tid; j <= U; j += NT) seg[j] = (uint16_t)(a.seg[j0 + j] - e0);
    for (int j = tid; j < U; j += NT) winv[j] = a.winv[j0 + j];
    for (int e = tid; e < 4 * k; e += NT) cval[e] = (uint16_t)(a.cval[e0 + e] - 4 * s0);
    Gp::sync();
    // a row's entries: the four vertices' stencil lists (ascending) merged
    auto walk = [&](int t, auto emit) {
        const ushort4 v = vidx[t];
        const int vs[4] = {v.x, v.y, v.z, v.w};
        int at[4], end[4], cur[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            at[q] = seg[vs[q]];
            end[q] = seg[vs[q] + 1];
            cur[q] = at[q] < end[q] ? cval[at[q]] : 0x7fffffff;
        }
        int n = 0;
        while (true) {
            const int c = min(min(cur[0] >> 2, cur[1] >> 2), min(cur[2] >> 2, cur[3] >> 2));
            if (c >= k) break;  // past every list's end
            float w = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if ((cur[q] >> 2) != c) continue;
                w += (q ? -1.0f / 3.0f : 1.0f) * ((cur[q] & 3) ? -1.0f / 3.0f : 1.0f) * winv[vs[q]];
                ++at[q];
                cur[q] = at[q] < end[q] ? cval[at[q]] : 0x7fffffff;
            }
            emit(n++, c, w);
        }
        return n;
    };
    // a row has at least the entries of its longest list: the rows of a hub, on
    // which merging is slow, are found too long before they are merged (700 rows
    // took 130 us to find it out, 1,300 half a millisecond)
#pragma unroll
    for (int v = 0; v < RPT; ++v) {
        const int t = tid + v * NT;
        int most = 0;
        if (t < k) {
            const ushort4 g = vidx[t];
            most = max(max(seg[g.x + 1] - seg[g.x], seg[g.y + 1] - seg[g.y]),
                       max(seg[g.z + 1] - seg[g.z], seg[g.w + 1] - seg[g.w]));
        }
        most = (int)__reduce_max_sync(0xffffffffu, (unsigned)most);
        if (lane == 0) sl[wq + v * (NT / 32)] = most;
    }
    Gp::sync();
    int least = 0;
    for (int q = 0; q < NS; ++q) least += sl[q];
    if (fixed - 64 + 256ll * least > bytes) return 1;
    Gp::sync();
    int off[RPT], len[RPT];
#pragma unroll
    for (int v = 0; v < RPT; ++v) {
        const int t = tid + v * NT;
        const int n = t < k ? walk(t, [](int, int, float) {}) : 0;
        len[v] = (int)__reduce_max_sync(0xffffffffu, (unsigned)n);
        if (lane == 0) sl[wq + v * (NT / 32)] = len[v];
    }
    Gp::sync();
    int total = 0;
#pragma unroll
    for (int v = 0; v < RPT; ++v) off[v] = 0;
    for (int q = 0; q < NS; ++q) {
#pragma unroll
        for (int v = 0; v < RPT; ++v)
            if (q == wq + v * (NT / 32)) off[v] = total;
        total += sl[q];
    }
    float2 *mat = (float2 *)(((uintptr_t)(sl + NS) + 15) & ~(uintptr_t)15);
    const long long used = (long long)((char *)mat - base) + 256ll * total;
    if (used > bytes) return 1;
    // u of the float64 residuals beside the matrix where it fits
    double *u64 = used + 24ll * U <= bytes ? (double *)(mat + 32 * total) : a.u64 + 3 * (size_t)j0;
#pragma unroll
    for (int v = 0; v < RPT; ++v) {
        const int t = tid + v * NT;
        float2 *m = mat + 32 * off[v] + lane;
        int n = 0;
        if (t < k) {
            const float4 nt4 = n4[t];
            n = walk(t, [&](int i, int c, float w) {
                const float4 b = n4[c];
                m[32 * i] = make_float2(w * (nt4.x * b.x + nt4.y * b.y + nt4.z * b.z), __int_as_float(c));
            });
        }
        for (int i = n; i < len[v]; ++i) m[32 * i] = make_float2(0.f, __int_as_float(0));
    }
    Gp::sync();  // the normals' place becomes r and z
    float r[RPT], x[RPT], p[RPT], s[RPT], w[RPT], zz[RPT];
    float4 pin[RPT];
    double lam[RPT];
    int blk[RPT];
#pragma unroll
    for (int v = 0; v < RPT; ++v) {
        const int t = tid + v * NT;
        const bool on = t < k;
        r[v] = on ? (float)a.b64[s0 + t] : 0.f;
        pin[v] = on ? a.pinv[s0 + t] : make_float4(0.f, 0.f, 0.f, 0.f);
        blk[v] = on ? grp[t] : 0;
        lam[v] = 0.0;
    }
    // one row per thread: its first entries in registers too
    constexpr int KEEP = RPT == 1 ? 8 : 0;
    float kv[KEEP + 1];
    int kc[KEEP + 1];
    if constexpr (KEEP > 0) {
#pragma unroll
        for (int i = 0; i < KEEP; ++i) {
            const float2 m = i < len[0] ? mat[32 * (off[0] + i) + lane] : make_float2(0.f, 0.f);
            kv[i] = m.x;
            kc[i] = __float_as_int(m.y);
        }
    }
    // z = P^-1 r and w = A z; the sums (r, z), (w, z), |r|^2
    auto apply = [&](float &ga, float &de, float &rh) {
#pragma unroll
        for (int v = 0; v < RPT; ++v)
            if (tid + v * NT < k) rS[tid + v * NT] = r[v];
        Gp::sync();
#pragma unroll
        for (int v = 0; v < RPT; ++v) {
            const int b0 = blk[v] >> 3, m = blk[v] & 7;
            float q = 0.f;
            if (m > 0) q = pin[v].x * rS[b0];
            if (m > 1) q += pin[v].y * rS[b0 + 1];
            if (m > 2) q += pin[v].z * rS[b0 + 2];
            if (m > 3) q += pin[v].w * rS[b0 + 3];
            zz[v] = q;
            if (m > 0) zS[tid + v * NT] = q;
        }
        Gp::sync();
        float g = 0.f, d = 0.f, h = 0.f;
#pragma unroll
        for (int v = 0; v < RPT; ++v) {
            const float2 *m = mat + 32 * off[v] + lane;
            float acc0 = 0.f, acc1 = 0.f, acc2 = 0.f, acc3 = 0.f;
            if constexpr (KEEP > 0) {
#pragma unroll
                for (int i = 0; i < KEEP; i += 4) {
                    acc0 += kv[i] * zS[kc[i]];
                    acc1 += kv[i + 1] * zS[kc[i + 1]];
                    acc2 += kv[i + 2] * zS[kc[i + 2]];
                    acc3 += kv[i + 3] * zS[kc[i + 3]];
                }
            }
            int i = KEEP;
            for (; i + 4 <= len[v]; i += 4) {
                const float2 m0 = m[32 * i], m1 = m[32 * (i + 1)], m2 = m[32 * (i + 2)], m3 = m[32 * (i + 3)];
                acc0 += m0.x * zS[__float_as_int(m0.y)];
                acc1 += m1.x * zS[__float_as_int(m1.y)];
                acc2 += m2.x * zS[__float_as_int(m2.y)];
                acc3 += m3.x * zS[__float_as_int(m3.y)];
            }
            for (; i < len[v]; ++i) {
                const float2 m0 = m[32 * i];
                acc0 += m0.x * zS[__float_as_int(m0.y)];
            }
            w[v] = (acc0 + acc1) + (acc2 + acc3);
            g += r[v] * zz[v];
            d += w[v] * zz[v];
            h += r[v] * r[v];
        }
        Gp::sum3h(g, d, h, red, ga, de, rh);
    };
    const double target = a.rel_tol * a.rel_tol * bb, third = 1.0 / 3.0;
    double rr = bb;
    int its = 0, rounds = 0;
    bool hand_over = false;
    const bool may_switch = BLK && a.block_switch > 0 && a.block_switch < a.maxit;
    const int cap_it = may_switch ? a.block_switch : a.maxit;
    while (rr > target && rounds < a.max_refine) {
#pragma unroll
        for (int v = 0; v < RPT; ++v) x[v] = p[v] = s[v] = 0.f;
        float gamma, delta, rho;
        apply(gamma, delta, rho);
        const float stop = (float)a.tol * (float)a.tol * rho;
        float alpha = gamma / delta, beta = 0.f;
        int it = 0;
        while (it < cap_it && rho > stop && rho > 0.f && alpha > 0.f && isfinite(alpha)) {
            // beta = g' / g and alpha' = g' / (d' - g' g' / (g alpha)): two
            // divisions deep, and rounded ones (a product with 1 / g would
            // overflow where g' / g does not)
            const float ga = gamma * alpha;
#pragma unroll
            for (int v = 0; v < RPT; ++v) {
                p[v] = zz[v] + beta * p[v];
                s[v] = w[v] + beta * s[v];
                x[v] += alpha * p[v];
                r[v] -= alpha * s[v];
            }
            float gn, dn, rn;
            apply(gn, dn, rn);
            beta = gn / gamma;
            alpha = gn / (dn - gn * (gn / ga));
            gamma = gn;
            rho = rn;
            ++it;
        }
        its += it;
        // lambda += x, then the float64 residual b - J M^-1 J^T lambda
#pragma unroll
        for (int v = 0; v < RPT; ++v) {
            lam[v] += (double)x[v];
            if (tid + v * NT < k) {
                lamS[2 * (tid + v * NT)] = lam[v];
                lamS[2 * (tid + v * NT) + 1] = -third * lam[v];
            }
        }
        Gp::sync();
        for (int j = tid; j < U; j += NT) {
            double a0 = 0.0, a1 = 0.0, a2 = 0.0;
            const int e1 = seg[j + 1];
            for (int e = seg[j]; e < e1; e += 4) {  // four entries' normals in flight
                double4_32a n[4];
                double p[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int c = cval[min(e + q, e1 - 1)];
                    n[q] = a.n64[s0 + (c >> 2)];
                    p[q] = lamS[2 * (c >> 2) + ((c & 3) ? 1 : 0)];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (e + q >= e1) break;
                    a0 += p[q] * n[q].x;
                    a1 += p[q] * n[q].y;
                    a2 += p[q] * n[q].z;
                }
            }
            const double wj = (double)winv[j];
            u64[3 * j] = wj * a0;
            u64[3 * j + 1] = wj * a1;
            u64[3 * j + 2] = wj * a2;
        }
        Gp::sync();
        double sum = 0.0;
        float rn[RPT];
#pragma unroll
        for (int v = 0; v < RPT; ++v) {
            const int t = tid + v * NT;
            rn[v] = 0.f;
            if (t >= k) continue;
            const ushort4 g = vidx[t];
            const double *ux = u64 + 3 * g.x, *ua = u64 + 3 * g.y, *ub = u64 + 3 * g.z, *uc = u64 + 3 * g.w;
            const double4_32a n = a.n64[s0 + t];
            const double d0 = ux[0] - (ua[0] + ub[0] + uc[0]) * third;
            const double d1 = ux[1] - (ua[1] + ub[1] + uc[1]) * third;
            const double d2 = ux[2] - (ua[2] + ub[2] + uc[2]) * third;
            const double q = a.b64[s0 + t] - (n.x * d0 + n.y * d1 + n.z * d2);
            rn[v] = (float)q;
            sum += q * q;
        }
        const double rr_new = Gp::sum(sum, redd);
        ++rounds;
        if (!(rr_new < rr)) {
            // the run did not reduce the float64 residual (a stagnating or
            // failing float32 run): its correction is taken back, the zone
            // keeps the best lambda found
#pragma unroll
            for (int v = 0; v < RPT; ++v) lam[v] -= (double)x[v];
            break;
        }
        const bool weak = rr_new * (ROWS_WEAK * ROWS_WEAK) > rr;
        rr = rr_new;
        if (weak && rr > ROWS_WEAK * ROWS_WEAK * target && rescue_fits(k, U, RESCUE_SMEM)) break;
#pragma unroll
        for (int v = 0; v < RPT; ++v) r[v] = rn[v];
        if (may_switch && it >= cap_it && rr > target) {
            hand_over = true;
            break;
        }
    }
#pragma unroll
    for (int v = 0; v < RPT; ++v)
        if (tid + v * NT < k) a.lam[s0 + tid + v * NT] = lam[v];
    res.rr = rr;
    res.its = its;
    res.rounds = rounds;
    return hand_over ? 2 : 0;
}

__device__ __forceinline__ void zone_finish(const ZoneArgs &a, int z, double rr, double bb, int its,
                                            int rounds, bool in_smem) {
    a.zres[z] = rr;
    a.zbb[z] = bb;
    atomicAdd(&a.ctl[1], its);
    atomicAdd(&a.ctl[2], rounds);
    atomicMax(&a.ctl[3], rounds);
    atomicOr(&a.ctl[4], in_smem ? 1 : 2);
}

// One warp per zone of at most WARP_ZONE stencils (most zones of a batch of
// small mesh pairs): a 256-thread CTA runs eight of them side by side, each
// in its own WARP_ZONE_SMEM slice of shared memory.
constexpr int WARP_ZONE = 32;
constexpr int WARP_ZONE_SMEM = 6272;  // at least zone_smem_need(32, 128, 32), a multiple of 16 B
constexpr int WARP_ZONE_WARPS = 8;

__global__ void __launch_bounds__(256, 4) k_cg_zone_warp(const int *d_nz, ZoneArgs a) {
    HFCR_PDL_WAIT();
    extern __shared__ float4 smem4[];
    const int nz = *d_nz, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    char *base = (char *)smem4 + (size_t)w * WARP_ZONE_SMEM;
    const int nwarps = gridDim.x * WARP_ZONE_WARPS;
    for (int z = blockIdx.x * WARP_ZONE_WARPS + w; z < nz; z += nwarps) {
        const int s0 = a.zs[z], k = a.zs[z + 1] - s0;
        if (k > WARP_ZONE) continue;
        const double bb = zone_start<WarpGroup>(a, s0, k, nullptr);
        ZoneResult r;
        if (solve_zone_rows<WarpGroup, 1, false>(a, z, base, WARP_ZONE_SMEM, bb, nullptr, nullptr, r)) {
            __syncwarp();
            r = solve_zone_smem<WarpGroup>(a, z, base, bb, nullptr, nullptr);
        }
        if (lane == 0) zone_finish(a, z, r.rr, bb, r.its, r.rounds, true);
        __syncwarp();  // the slice is reused by the warp's next zone
    }
}

// Zone z solved by the thread group Gp: staged in shared memory at base
// when its data fit smem_bytes, else the same rounds on global scratch.
// The two paths are instantiated separately so that the shared-memory one
// sees pointers derived only from the shared array (LDS/STS, not generic
// loads).
struct ZoneScratch {
    float *x, *r, *p, *s, *w, *z, *u;
};

// RPT: rows per thread of the solver by rows, tried first (0: never)
template <class Gp, int RPT, bool BLK = false>
__device__ __forceinline__ void solve_zone(const ZoneArgs &a, int z, char *base, int smem_bytes,
                                           float *red, double *redd, const ZoneScratch &g) {
    const int tid = Gp::rank(), nt = Gp::size();
    const int s0 = a.zs[z], k = a.zs[z + 1] - s0;
    const int j0 = a.zv[z], U = a.zv[z + 1] - j0;
    const double bb = zone_start<Gp>(a, s0, k, redd);
    const int g0 = a.zg[z], G = a.zg[z + 1] - g0;
    const bool in_smem = zone_smem_need(k, U, G) <= smem_bytes;
    int its = 0, rounds = 0;
    double rr;
    ZoneResult first;
    int how = 1;
    if constexpr (RPT > 0) {
        how = solve_zone_rows<Gp, RPT, BLK>(a, z, base, smem_bytes, bb, red, redd, first);
        Gp::sync();  // shared memory is the next solver's
    }
    if (how == 0) {
        rr = first.rr;
        its = first.its;
        rounds = first.rounds;
    } else if (in_smem) {
        const ZoneResult r = solve_zone_smem<Gp, BLK>(a, z, base, bb, red, redd, how == 2 ? &first : nullptr);
        rr = r.rr;
        its = r.its;
        rounds = r.rounds;
    } else {
        const double target = a.rel_tol * a.rel_tol * bb;
        CgView v;
        v.r = g.r + s0; v.p = g.p + s0; v.x = g.x + s0; v.sv = g.s + s0; v.w = g.w + s0;
        v.z = g.z + s0;
        v.u = (float4 *)g.u + j0;
        v.n4 = a.n32 + s0;
        v.pinv = a.pinv + s0; v.gst = a.gst + g0; v.G = G; v.goff = s0;
        v.vidx = a.vidx + s0; v.seg = a.seg + j0; v.cval = a.cval; v.winv = a.winv + j0;
        v.voff = j0; v.coff = 4 * s0; v.eoff = 0;
        for (int t = tid; t < k; t += nt) v.r[t] = (float)a.b64[s0 + t];
        rr = bb;
        while (rr > target && rounds < a.max_refine) {
            for (int t = tid; t < k; t += nt) {
                v.p[t] = 0.f;
                v.sv[t] = 0.f;
                v.x[t] = 0.f;
            }
            Gp::sync();
            its += cg_cg_loop<Gp>(v, k, U, a.maxit, (float)a.tol, red);
            for (int t = tid; t < k; t += nt) a.lam[s0 + t] += (double)v.x[t];
            Gp::sync();
            const double rr_prev = rr;
            rr = zone_residual<Gp>(v, k, U, s0, j0, a.n64, a.b64, a.lam, a.u64, redd);
            ++rounds;
            if (!(rr < rr_prev)) {  // as in the staged path: the run is taken back
                for (int t = tid; t < k; t += nt) a.lam[s0 + t] -= (double)v.x[t];
                rr = rr_prev;
                Gp::sync();
                break;
            }
        }
    }
    if (tid == 0) zone_finish(a, z, rr, bb, its, rounds, how == 0 || in_smem);
    Gp::sync();  // shared memory is reused by the group's next zone
}

// The mixed solver's CTA launches (k_cg_zone_warp takes the zones of at
// most WARP_ZONE stencils).  k_cg_zone_pair: the zones of ZONE_MID to
// ZONE_BIG - 1 stencils one at a time on all 512 threads, then the smaller
// ones two at a time, one per 256-thread half (its own named barrier, half
// the shared memory), so that a zone gets about one to four rows per
// thread.  k_cg_zone<BIG_ZONE_THREADS>: the rest, one CTA with all of
// shared memory each (512 threads: measured a little faster than 1,024 on
// the frame sequence's large zones, 0.546 against 0.566 ms per frame, and
// cheaper barriers and reductions).  (solve_zone
// ends with its group's barrier, so the halves may reuse the shared memory
// of the CTA's last whole-CTA zone.)
// Zone assignment of the pair launch: a solver's first zone is fixed (so
// that while there are fewer zones than solvers each zone has an SM to
// itself), the following ones are taken from a counter in turn (zones
// differ widely in size; the counter balances them).  stride = the
// solvers; the counter counts the zones taken beyond the fixed ones.
// Returns the group's next zone, identical in every thread of the group
// (slot: the group's shared word).
template <class Gp>
__device__ __forceinline__ int next_zone(unsigned *counter, int stride, int *slot) {
    if (Gp::rank() == 0) *slot = stride + (int)atomicAdd(counter, 1u);
    Gp::sync();
    const int z = *slot;
    Gp::sync();  // the slot is rewritten by the next call
    return z;
}

// The zones of at least ZONE_MID stencils go to the large-zone launch, one
// CTA each, when at least one of them has ZONE_BIG stencils or more and
// there are at most ROUTE_MAX of them (and no more than its CTAs): a
// frame's large contact zone and the few medium ones beside it then run
// side by side instead of one launch after the other, and each may switch
// to its blocks.  Otherwise the pair launch takes those below ZONE_BIG:
// alone, a medium zone is faster there (measured: a 538-row zone of the
// two-tori scene, 0.26 against 0.37 ms; the large-zone CTA's shared memory
// leaves little L1 for the float64 rounds), and many of them (a batch)
// share its two CTAs per SM.  Both launches count the zones from the zone
// starts (one barrier per blockDim.x zones), so they take the same
// decision.  Returns how many zones have at least lo stencils, *n_big how
// many at least ZONE_BIG; *pick: the zone of rank `rank` among the first
// ones in zone order, -1 if none (all identical in every thread of the CTA).
constexpr int ROUTE_MAX = 8;

__device__ __forceinline__ int zones_at_least(const int *zs, int nz, int lo, int rank, int *pick,
                                              int *n_big) {
    __shared__ int wc[32];
    __shared__ int found;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) found = -1;
    int total = 0, big = 0;
    for (int base = 0; base < nz; base += blockDim.x) {
        const int z = base + threadIdx.x;
        const int kz = z < nz ? zs[z + 1] - zs[z] : 0;
        const bool pred = kz >= lo;
        big += __syncthreads_count(kz >= ZONE_BIG);
        const int c = __syncthreads_count(pred);
        if (rank >= total && rank < total + c) {  // the same in every thread
            const unsigned bal = __ballot_sync(0xffffffffu, pred);
            if (lane == 0) wc[w] = __popc(bal);
            __syncthreads();
            int before = total + __popc(bal & ((1u << lane) - 1u));
            for (int q = 0; q < w; ++q) before += wc[q];
            if (pred && before == rank) found = z;
        }
        total += c;
    }
    __syncthreads();
    *pick = found;
    *n_big = big;
    return total;
}

// the zones of small_lo < k < ZONE_MID stencils on half H (first fixed
// zone: blockIdx.x + H gridDim.x)
template <int H>
__device__ __forceinline__ void half_zones(const ZoneArgs &a, int nz, int small_lo, char *base,
                                           int bytes, float *red, double *redd,
                                           const ZoneScratch &g, int *slot) {
    const bool more = nz > 2 * (int)gridDim.x;  // zones beyond the fixed ones
    for (int z = blockIdx.x + H * gridDim.x; z < nz;
         z = more ? next_zone<HalfGroup<H>>(a.ticket + 1, 2 * gridDim.x, slot) : nz) {
        const int k = a.zs[z + 1] - a.zs[z];
        if (k <= small_lo || k >= ZONE_MID) continue;
        solve_zone<HalfGroup<H>, 1>(a, z, base, bytes, red, redd, g);
    }
}

__global__ void __launch_bounds__(512, 2) k_cg_zone_pair(const int *d_nz, ZoneArgs a, int small_lo,
                                                         ZoneScratch g, int smem_bytes, int big_ctas) {
    HFCR_PDL_WAIT();
    extern __shared__ float4 smem4[];
    __shared__ float red[96];     // halves: 32 floats each; the whole CTA: 64
    __shared__ double redd[16];   // halves: 8 each; the whole CTA: 16
    __shared__ int slot[3];
    const int nz = *d_nz;
    // the larger zones first, on all 512 threads (unless the large-zone
    // launch takes them)
    __shared__ int first;
    {
        int unused, n_big;
        const int n_mid = zones_at_least(a.zs, nz, ZONE_MID, -1, &unused, &n_big);
        const bool to_big = n_big > 0 && n_mid <= ROUTE_MAX && n_mid <= big_ctas;
        if (threadIdx.x == 0) first = to_big ? nz : (int)blockIdx.x;
        __syncthreads();
    }
    const bool more = nz > (int)gridDim.x;  // zones beyond the fixed ones
    for (int z = first; z < nz; z = more ? next_zone<CtaGroup>(a.ticket, gridDim.x, slot + 2) : nz) {
        const int k = a.zs[z + 1] - a.zs[z];
        if (k < ZONE_MID || k >= ZONE_BIG) continue;
        solve_zone<CtaGroup, 2>(a, z, (char *)smem4, smem_bytes, red, redd, g);
    }
    // then the smaller ones, two at a time (a whole-CTA zone ends with a
    // barrier of the whole CTA, so the halves may reuse the shared memory)
    const int half_bytes = (smem_bytes / 2) & ~15;
    if (threadIdx.x < 256)
        half_zones<0>(a, nz, small_lo, (char *)smem4, half_bytes, red, redd, g, slot);
    else
        half_zones<1>(a, nz, small_lo, (char *)smem4 + half_bytes, half_bytes, red + 32, redd + 8,
                      g, slot + 1);
}

// The zones of more than k_lo stencils, one CTA each; or, when the zones
// of at least mid_lo stencils come to this launch (zones_at_least), the
// zone of rank blockIdx.x among those.  leave_big: zones that do not
// fit smem_bytes are left to the cluster solver (k_cg_zone_cl) instead of
// the global-memory path.
template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1) k_cg_zone(const int *d_nz, ZoneArgs a, int k_lo,
                                                        int mid_lo, ZoneScratch g, int smem_bytes,
                                                        int leave_big) {
    HFCR_PDL_WAIT();
    extern __shared__ float4 smem4[];
    __shared__ float red[96];
    __shared__ double redd[THREADS / 32];
    const int nz = *d_nz;
    // the loop's first zone, its stride, and the zones' smallest size minus one
    __shared__ int sel[3];
    {
        int pick, n_big;
        const int n_mid = zones_at_least(a.zs, nz, mid_lo, blockIdx.x, &pick, &n_big);
        const bool ranked = n_big > 0 && n_mid <= ROUTE_MAX && n_mid <= (int)gridDim.x;
        if (threadIdx.x == 0) {
            sel[0] = ranked ? (pick >= 0 ? pick : nz) : (int)blockIdx.x;
            sel[1] = ranked ? nz : (int)gridDim.x;
            sel[2] = ranked ? mid_lo - 1 : k_lo;
        }
        __syncthreads();
    }
    for (int z = sel[0]; z < nz; z += sel[1]) {
        const int k = a.zs[z + 1] - a.zs[z];
        if (k <= sel[2]) continue;
        if (leave_big && zone_smem_need(k, a.zv[z + 1] - a.zv[z], a.zg[z + 1] - a.zg[z]) > smem_bytes)
            continue;
        solve_zone<CtaGroup, 3, true>(a, z, (char *)smem4, smem_bytes, red, redd, g);
        if (threadIdx.x == 0) {  // rows and touched vertices of the zones of this launch
            atomicAdd(&a.ctl[5], k);
            atomicAdd(&a.ctl[6], a.zv[z + 1] - a.zv[z]);
        }
    }
}

// ---------------------------------------------------------------------------
// The plain float64 form's per-zone solve: the same impact zones,
// zone-ordered rows, vertex CSR and block-Jacobi groups as the mixed
// solver, each zone solved by one 256-thread CTA with preconditioned CG in
// the Chronopoulos-Gear form, in float64 on the float64 normals, on global
// (L2-resident) arrays, to |r_zone| <= rel_tol |b_zone| (no refinement: the
// arithmetic is already float64).
// ---------------------------------------------------------------------------

struct Zone64Scratch {
    double *r, *p, *s, *w, *z;  // [cap_k] each, zone-ordered rows
};

constexpr int ZONE64_THREADS = 256;

// three block sums with one barrier, identical in every thread (the
// float64 counterpart of block_sum3)
__device__ __forceinline__ void block_sum3d(double a, double b, double c, double *red, double &sa,
                                            double &sb_, double &sc) {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();  // red is free of its previous use
    if (lane == 0) {
        red[3 * w] = a;
        red[3 * w + 1] = b;
        red[3 * w + 2] = c;
    }
    __syncthreads();
    const int nw = blockDim.x >> 5;
    double x = lane < nw ? red[3 * lane] : 0.0;
    double y = lane < nw ? red[3 * lane + 1] : 0.0;
    double q = lane < nw ? red[3 * lane + 2] : 0.0;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
        q += __shfl_xor_sync(0xffffffffu, q, o);
    }
    sa = __shfl_sync(0xffffffffu, x, 0);
    sb_ = __shfl_sync(0xffffffffu, y, 0);
    sc = __shfl_sync(0xffffffffu, q, 0);
}

// out = J M^-1 J^T in over the zone's rows (u: the zone's touched
// vertices, 3 doubles each); returns nothing, the caller synchronises
__device__ __forceinline__ void zone64_vertex(const ZoneArgs &a, int s0, int j0, int U,
                                              const double *in, double *u) {
    const double third = 1.0 / 3.0;
    for (int j = threadIdx.x; j < U; j += blockDim.x) {
        double a0 = 0.0, a1 = 0.0, a2 = 0.0;
        for (int e = a.seg[j0 + j]; e < a.seg[j0 + j + 1]; ++e) {
            const int c = a.cval[e] - 4 * s0;
            const int sl = c >> 2;
            const double ps = ((c & 3) ? -third : 1.0) * in[sl];
            const double4_32a n = a.n64[s0 + sl];
            a0 += ps * n.x;
            a1 += ps * n.y;
            a2 += ps * n.z;
        }
        const double wv = (double)a.winv[j0 + j];
        u[3 * j] = wv * a0;
        u[3 * j + 1] = wv * a1;
        u[3 * j + 2] = wv * a2;
    }
}

__device__ __forceinline__ double zone64_stencil(const ZoneArgs &a, int s0, int j0, int t,
                                                 const double *u) {
    const double third = 1.0 / 3.0;
    const int4 g = a.vidx[s0 + t];
    const double *ux = u + 3 * (g.x - j0), *ua = u + 3 * (g.y - j0), *ub = u + 3 * (g.z - j0),
                 *uc = u + 3 * (g.w - j0);
    const double4_32a n = a.n64[s0 + t];
    return n.x * (ux[0] - (ua[0] + ub[0] + uc[0]) * third) +
           n.y * (ux[1] - (ua[1] + ub[1] + uc[1]) * third) +
           n.z * (ux[2] - (ua[2] + ub[2] + uc[2]) * third);
}

// z = P^-1 r over the zone's groups (the float64 inverse blocks)
__device__ __forceinline__ void zone64_precond(const ZoneArgs &a, int s0, int g0, int G,
                                               const double *r, double *zz) {
    for (int gi = threadIdx.x; gi < G; gi += blockDim.x) {
        const int lo = a.gst[g0 + gi] - s0, hi = a.gst[g0 + gi + 1] - s0;
        double rr[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) rr[q] = lo + q < hi ? r[lo + q] : 0.0;
        for (int t = lo; t < hi; ++t) {
            const double4_32a m = a.pinv64[s0 + t];
            zz[t] = m.x * rr[0] + m.y * rr[1] + m.z * rr[2] + m.w * rr[3];
        }
    }
}

// A zone's float64 CG with everything an iteration touches in shared memory
// and the rows' vectors in registers.  float64 runs at two lanes per clock and
// SM, half a lane in each quarter: a warp's operation takes 64 cycles, a
// division about a thousand, and an iteration is a chain of them.  So a
// warp's sums are halved, warps without rows or vertices take no part, and one
// warp forms the step's scalars for all, the reciprocals of the step before
// while the others update their rows.  Products stay J M^-1 (J^T z): with the
// merged matrix of solve_zone_rows an iteration was a quarter shorter, but
// the rounding of its entries cost an ill-conditioned zone two digits of dx.
// An iteration sums over the tree of the float64 solver's RESCUE_NT threads and
// divides as it does (the unstaged form below has twice the threads, hence
// another tree).  A zone of 97 rows (93 iterations) 853 -> 584 us, one of 354
// rows (75) 1,175 -> 835.  False when the zone does not fit (nothing done);
// otherwise lambda is stored and the count in its.
constexpr int RESCUE_THREADS = 512;
constexpr int RESCUE_VT = RESCUE_THREADS - 32;  // threads with vertices

// a / b rounded to nearest from y = 1 / b rounded to nearest.  a y is off by up to
// 1.5 ulp; corrected by its residual it is within an ulp, and from there the
// second correction is a / b rounded to nearest (Markstein 1990, which asks for
// such a start).  Results and residuals that may be subnormal divide instead.
__device__ __forceinline__ double div_by(double a, double b, double y) {
    const double q = a * y, f = fma(fma(-b, q, a), y, q), c = fma(fma(-b, f, a), y, f);
    return isfinite(q) && fabs(q) > 1e-280 && fabs(a) > 1e-280 ? c : a / b;
}

__device__ __forceinline__ double warp_halve3d(double a, double b, double c) {  // as warp_halve3
    const int lane = threadIdx.x & 31;
    const bool h = lane & 16, q = lane & 8;
    const double x = (h ? c : a) + __shfl_xor_sync(0xffffffffu, h ? a : c, 16);
    const double y = (h ? 0.0 : b) + __shfl_xor_sync(0xffffffffu, h ? b : 0.0, 16);
    double t = (q ? y : x) + __shfl_xor_sync(0xffffffffu, q ? x : y, 8);
#pragma unroll
    for (int o = 4; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

__device__ __forceinline__ bool zone64_staged(const ZoneArgs &a, int z, char *base, int bytes, double bb,
                                              int maxit, double *red, double *sc, int &its) {
    constexpr int NT = RESCUE_NT, RPT = RESCUE_ROWS;
    static_assert(NT == 256 && NT == ZONE64_THREADS && RESCUE_VT == 480, "the named barriers below; eight warps' sums");
    const int tid = threadIdx.x, lane = tid & 31, wq = tid >> 5;
    const int s0 = a.zs[z], k = a.zs[z + 1] - s0;
    const int j0 = a.zv[z], U = a.zv[z + 1] - j0;
    const int g0 = a.zg[z], G = a.zg[z + 1] - g0;
    const int e0 = a.seg[j0];
    // layout: blocks' inverse rows | normals | z, -z / 3 | r | u | vidx | winv | seg | cval | groups
    if (!rescue_fits(k, U, bytes)) return false;
    double4_32a *pS = (double4_32a *)base;
    double *nS = (double *)(pS + k), *zS = nS + 3 * k, *rS = zS + 2 * k, *uS = rS + k;
    ushort4 *vidx = (ushort4 *)(uS + 3 * U);
    float *winv = (float *)(vidx + k);
    uint16_t *seg = (uint16_t *)(winv + U);
    uint16_t *cval = seg + U + 1;
    uint16_t *grp = cval + 4 * k;
    const double third = 1.0 / 3.0;
    for (int t = tid; t < k; t += RESCUE_THREADS) {
        const int4 g = a.vidx[s0 + t];
        vidx[t] = make_ushort4((unsigned short)(g.x - j0), (unsigned short)(g.y - j0),
                               (unsigned short)(g.z - j0), (unsigned short)(g.w - j0));
        const double4_32a n = a.n64[s0 + t];
        nS[3 * t] = n.x;
        nS[3 * t + 1] = n.y;
        nS[3 * t + 2] = n.z;
        pS[t] = a.pinv64[s0 + t];
    }
    for (int g = tid; g < G; g += RESCUE_THREADS) {  // each row's block: first row and size
        const int b0 = a.gst[g0 + g] - s0, b1 = a.gst[g0 + g + 1] - s0;
        for (int t = b0; t < b1; ++t) grp[t] = (uint16_t)(b0 << 3 | (b1 - b0));
    }
    for (int j = tid; j <= U; j += RESCUE_THREADS) seg[j] = (uint16_t)(a.seg[j0 + j] - e0);
    for (int j = tid; j < U; j += RESCUE_THREADS) winv[j] = a.winv[j0 + j];
    for (int e = tid; e < 4 * k; e += RESCUE_THREADS) cval[e] = (uint16_t)(a.cval[e0 + e] - 4 * s0);
    __syncthreads();
    its = 0;
    if (tid >= RESCUE_VT) {
        const double stop = a.rel_tol * a.rel_tol * bb;
        double gamma = 1.0, alpha = 1.0, rg = 1.0, ra = 1.0;  // of the step before, and their reciprocals
        for (bool first = true;; first = false) {
            __syncthreads();  // the warps' sums
            double t = red[4 * (lane & 7) + (lane >> 3)];
#pragma unroll
            for (int o = 4; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            const double gn = __shfl_sync(0xffffffffu, t, 0), dn = __shfl_sync(0xffffffffu, t, 8),
                         rn = __shfl_sync(0xffffffffu, t, 16);
            double beta = 0.0;
            if (first) {
                alpha = gn / dn;
            } else {
                beta = div_by(gn, gamma, rg);
                alpha = gn / (dn - div_by(beta * gn, alpha, ra));
            }
            const bool go = its < maxit && rn > stop && alpha > 0.0 && isfinite(alpha);
            if (lane == 0) {
                sc[0] = alpha;
                sc[1] = beta;
                *(int *)(sc + 2) = go;
            }
            __syncthreads();
            if (!go) break;
            ++its;
            gamma = gn;
            rg = 1.0 / gn;
            ra = 1.0 / alpha;
        }
    } else {
        double r[RPT], x[RPT], p[RPT], s[RPT], w[RPT], zz[RPT];
        const bool rows = tid < NT;
#pragma unroll
        for (int v = 0; v < RPT; ++v) {
            const int t = tid + v * NT;
            r[v] = rows && t < k ? a.b64[s0 + t] : 0.0;
            x[v] = p[v] = s[v] = w[v] = zz[v] = 0.0;
        }
        while (true) {
            if (rows) {  // z = P^-1 r
#pragma unroll
                for (int v = 0; v < RPT; ++v)
                    if (tid + v * NT < k) rS[tid + v * NT] = r[v];
                asm volatile("bar.sync 1, 256;" ::: "memory");
#pragma unroll
                for (int v = 0; v < RPT; ++v) {
                    const int t = tid + v * NT;
                    if (t >= k) continue;
                    const int b0 = grp[t] >> 3, m = grp[t] & 7;
                    double rr[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) rr[q] = q < m ? rS[b0 + q] : 0.0;
                    const double4_32a pi = pS[t];
                    zz[v] = pi.x * rr[0] + pi.y * rr[1] + pi.z * rr[2] + pi.w * rr[3];
                    zS[2 * t] = zz[v];
                    zS[2 * t + 1] = -third * zz[v];
                }
            }
            asm volatile("bar.sync 2, 480;" ::: "memory");
            for (int j = tid; j < U; j += RESCUE_VT) {  // u = M^-1 J^T z
                double a0 = 0.0, a1 = 0.0, a2 = 0.0;
                const int e1 = seg[j + 1];
#pragma unroll 2
                for (int e = seg[j]; e < e1; ++e) {
                    const int c = cval[e], sl = c >> 2;
                    const double ps = zS[2 * sl + ((c & 3) ? 1 : 0)];
                    a0 += ps * nS[3 * sl];
                    a1 += ps * nS[3 * sl + 1];
                    a2 += ps * nS[3 * sl + 2];
                }
                const double wv = (double)winv[j];
                uS[3 * j] = wv * a0;
                uS[3 * j + 1] = wv * a1;
                uS[3 * j + 2] = wv * a2;
            }
            asm volatile("bar.sync 2, 480;" ::: "memory");
            if (rows) {  // w = J u and the sums (r, z), (w, z), |r|^2
                double t = 0.0;
                if (wq * 32 < k) {
                    double g = 0.0, d = 0.0, h = 0.0;
#pragma unroll
                    for (int v = 0; v < RPT; ++v) {
                        const int t = tid + v * NT;
                        if (t >= k) continue;
                        const ushort4 i = vidx[t];
                        const double *ux = uS + 3 * i.x, *ua = uS + 3 * i.y, *ub = uS + 3 * i.z, *uc = uS + 3 * i.w;
                        const double nx = nS[3 * t], ny = nS[3 * t + 1], nz = nS[3 * t + 2];
                        w[v] = nx * (ux[0] - (ua[0] + ub[0] + uc[0]) * third) +
                               ny * (ux[1] - (ua[1] + ub[1] + uc[1]) * third) +
                               nz * (ux[2] - (ua[2] + ub[2] + uc[2]) * third);
                        g += r[v] * zz[v];
                        d += w[v] * zz[v];
                        h += r[v] * r[v];
                    }
                    t = warp_halve3d(g, d, h);
                }
                if ((lane & 7) == 0) red[4 * wq + (lane >> 3)] = t;
            }
            __syncthreads();
            __syncthreads();  // the scalars
            if (!*(volatile int *)(sc + 2)) break;
            ++its;
            const double al = sc[0], be = sc[1];
            if (rows) {
#pragma unroll
                for (int v = 0; v < RPT; ++v) {
                    if (tid + v * NT >= k) continue;
                    p[v] = zz[v] + be * p[v];
                    s[v] = w[v] + be * s[v];
                    x[v] += al * p[v];
                    r[v] -= al * s[v];
                }
            }
        }
#pragma unroll
        for (int v = 0; v < RPT; ++v)
            if (rows && tid + v * NT < k) a.lam[s0 + tid + v * NT] = x[v];
    }
    __syncthreads();
    return true;
}

// RESCUE: only the zones whose recorded |r|^2 (the mixed solver's) misses
// the target, solved again from lam = 0 (zones on which the float32 runs
// stopped reducing the float64 residual), staged where they fit; otherwise
// every zone (several CTAs per SM), its vectors in global memory
template <bool RESCUE>
__global__ void __launch_bounds__(RESCUE ? RESCUE_THREADS : ZONE64_THREADS)
    k_cg_zone64(const int *d_nz, ZoneArgs a, Zone64Scratch g, int maxit, int smem_bytes) {
    HFCR_PDL_WAIT();
    extern __shared__ float4 smem4[];
    constexpr int WARPS = (RESCUE ? RESCUE_THREADS : ZONE64_THREADS) / 32;
    __shared__ double red[4 * WARPS];
    __shared__ double redd[WARPS];
    __shared__ double sc[3];
    const int nz = *d_nz;
    for (int z = blockIdx.x; z < nz; z += gridDim.x) {
        if (RESCUE && a.zres[z] <= a.rel_tol * a.rel_tol * a.zbb[z]) continue;
        const int s0 = a.zs[z], k = a.zs[z + 1] - s0;
        const int j0 = a.zv[z], U = a.zv[z + 1] - j0;
        const int g0 = a.zg[z], G = a.zg[z + 1] - g0;
        const double bb = zone_start<CtaGroup>(a, s0, k, redd);  // lam = 0 on the zone's rows
        // the zone's block-Jacobi inverses in float64 (a block of nearly
        // dependent rows has a large inverse that float32 would not hold)
        group_inverses<PlainLd>(g0, (int)(threadIdx.x >> 5), (int)(blockDim.x >> 5), g0 + G, a.gst,
                                a.ids, a.n64, a.nA, a.wA, a.wB, a.pinv64);
        __syncthreads();  // the blocks, read by other threads below
        double *r = g.r + s0, *p = g.p + s0, *sv = g.s + s0, *w = g.w + s0, *zz = g.z + s0;
        double *x = a.lam + s0, *u = a.u64 + 3 * (size_t)j0;
        int it = 0;
        bool staged = false;
        if constexpr (RESCUE) staged = zone64_staged(a, z, (char *)smem4, smem_bytes, bb, maxit, red, sc, it);
        if (!staged) {
            for (int t = threadIdx.x; t < k; t += blockDim.x) {
                r[t] = a.b64[s0 + t];
                p[t] = 0.0;
                sv[t] = 0.0;
            }
            __syncthreads();
            zone64_precond(a, s0, g0, G, r, zz);
            __syncthreads();
            zone64_vertex(a, s0, j0, U, zz, u);
            __syncthreads();
            double ga = 0.0, de = 0.0, rh = 0.0;
            for (int t = threadIdx.x; t < k; t += blockDim.x) {
                const double wt = zone64_stencil(a, s0, j0, t, u);
                w[t] = wt;
                ga += r[t] * zz[t];
                de += wt * zz[t];
                rh += r[t] * r[t];
            }
            double gamma, delta, rho;
            block_sum3d(ga, de, rh, red, gamma, delta, rho);
            const double stop = a.rel_tol * a.rel_tol * bb;
            double alpha = gamma / delta, beta = 0.0;
            it = 0;
            while (it < maxit && rho > stop && alpha > 0.0 && isfinite(alpha)) {
                for (int t = threadIdx.x; t < k; t += blockDim.x) {
                    const double pt = zz[t] + beta * p[t];
                    const double st = w[t] + beta * sv[t];
                    p[t] = pt;
                    sv[t] = st;
                    x[t] += alpha * pt;
                    r[t] -= alpha * st;
                }
                __syncthreads();
                zone64_precond(a, s0, g0, G, r, zz);
                __syncthreads();
                zone64_vertex(a, s0, j0, U, zz, u);
                __syncthreads();
                ga = de = rh = 0.0;
                for (int t = threadIdx.x; t < k; t += blockDim.x) {
                    const double wt = zone64_stencil(a, s0, j0, t, u);
                    w[t] = wt;
                    ga += r[t] * zz[t];
                    de += wt * zz[t];
                    rh += r[t] * r[t];
                }
                double gn, dn, rn;
                block_sum3d(ga, de, rh, red, gn, dn, rn);
                beta = gn / gamma;
                alpha = gn / (dn - beta * gn / alpha);
                gamma = gn;
                rho = rn;
                ++it;
            }
        }
        // the zone's true residual b - A lam (not the recurrence's)
        __syncthreads();
        zone64_vertex(a, s0, j0, U, x, u);
        __syncthreads();
        double rr = 0.0;
        for (int t = threadIdx.x; t < k; t += blockDim.x) {
            const double rt = a.b64[s0 + t] - zone64_stencil(a, s0, j0, t, u);
            rr += rt * rt;
        }
        rr = block_sum_uniform(rr, redd);
        if (threadIdx.x == 0) {
            a.zres[z] = rr;
            a.zbb[z] = bb;
            atomicAdd(&a.ctl[1], it);
            atomicAdd(&a.ctl[2], 1);
            atomicMax(&a.ctl[3], 1);
            atomicOr(&a.ctl[4], 4);
        }
        __syncthreads();  // u and the scalars' shared words are reused by the next zone
    }
}

// ---------------------------------------------------------------------------
// Large impact zones on a thread-block cluster: the zone's rows and touched
// vertices are split over the CL CTAs of a cluster (CL SMs), each CTA
// stages its share in its own shared memory, and the products that cross
// shares read the other CTAs' shared memory directly (distributed shared
// memory) between hardware cluster barriers.  The arithmetic is that of the
// one-CTA staged solve (float32 Chronopoulos-Gear PCG on the float32
// normals, block-Jacobi groups, float64 residual rounds, the same stopping
// rules); zones too large for one SM's shared memory (which would
// otherwise iterate on global memory) stay in shared memory, up to CL times
// larger.  (Measured: a zone that fits one SM iterates no faster on a
// cluster: an iteration is a chain of barriers and dependent loads either
// way, so such zones stay on one CTA.)  Rows are split at group boundaries, so
// the preconditioner stays local to a CTA.  Every CTA uses one layout,
// sized for the largest share of the zone, so another CTA's array is this
// CTA's array mapped to that rank.  Reductions: each CTA writes its
// partial sums into every CTA's slot for it, and after the barrier each
// CTA adds the CL slots in rank order (identical sums everywhere).
// ---------------------------------------------------------------------------

constexpr int CL = 8;               // CTAs per cluster (portable cluster size)
constexpr int CL_THREADS = 512;
constexpr int CL_SMEM = 200 * 1024; // dynamic shared memory per CTA
constexpr int ZONE_CL_MIN = ZONE_BIG;  // zones of at least this many rows

namespace cgx = cooperative_groups;

struct ClLayout {
    int Kc, Uc, Ec, Gc;       // capacities: rows, vertices, CSR entries, groups per CTA
    int o_n4, o_pinv, o_vidx, o_u, o_f, o_winv, o_seg, o_ent, o_gst;
    int bytes;
};

__device__ __forceinline__ ClLayout cl_layout(int Kc, int Uc, int Ec, int Gc) {
    ClLayout L;
    L.Kc = Kc; L.Uc = Uc; L.Ec = Ec; L.Gc = Gc;
    int o = 0;
    L.o_n4 = o;   o += 16 * Kc;
    L.o_pinv = o; o += 16 * Kc;
    L.o_vidx = o; o += 16 * Kc;
    L.o_u = o;    o += 16 * Uc;
    L.o_f = o;    o += 4 * 6 * Kc;          // r p x sv w z
    L.o_winv = o; o += 4 * Uc;
    L.o_seg = o;  o += 4 * (Uc + 1);
    L.o_ent = o;  o += 4 * Ec;
    L.o_gst = o;  o += 4 * (Gc + 1);
    L.bytes = o;
    return L;
}

// the partial sums of this CTA (nv values, the same in every thread) into
// slot `rank` of every CTA's red, then after the barrier the sums over the
// CL slots in rank order
template <typename T, int NV>
__device__ __forceinline__ void cl_reduce(cgx::cluster_group &cl, const T *part, T *red, T *out) {
    if (threadIdx.x < CL * NV) {
        const int dst = threadIdx.x / NV, v = threadIdx.x % NV;
        T *r = cl.map_shared_rank(red, dst);
        r[cl.block_rank() * NV + v] = part[v];
    }
    cl.sync();
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        T t = 0;
        for (int c = 0; c < CL; ++c) t += red[c * NV + v];
        out[v] = t;
    }
}

// CTA-wide float sums of three values (identical in every thread)
__device__ __forceinline__ void cl_block3(float a, float b, float c, float *red, float *out) {
    float sa, sb, sc;
    block_sum3(a, b, c, red, sa, sb, sc);
    __syncthreads();  // red is rewritten by the next call
    out[0] = sa; out[1] = sb; out[2] = sc;
}

// one_cta_smem: the shared memory of the one-CTA solver (k_cg_zone): the
// zones that fit it are its, this kernel takes the larger ones
__global__ void __launch_bounds__(CL_THREADS, 1) k_cg_zone_cl(const int *d_nz, ZoneArgs a,
                                                              ZoneScratch gs, int one_cta_smem) {
    HFCR_PDL_WAIT();
    cgx::cluster_group cl = cgx::this_cluster();
    extern __shared__ float4 smem4[];
    char *base = (char *)smem4;
    __shared__ float redf[CL * 3];          // cluster partials (float)
    __shared__ double redd[CL * 2];         // cluster partials (double)
    __shared__ float bred[96];              // block reductions
    __shared__ double bredd[CL_THREADS / 32];
    __shared__ int rb[CL + 1], gb[CL + 1], vb[CL + 1], eb[CL + 1];
    const int rank = cl.block_rank();
    const int tid = threadIdx.x, nt = CL_THREADS;
    const int nz = *d_nz;
    const int ncl = gridDim.x / CL;
    const int ci = blockIdx.x / CL;
    for (int z = ci; z < nz; z += ncl) {
        const int s0 = a.zs[z], k = a.zs[z + 1] - s0;
        if (k < ZONE_CL_MIN) continue;
        const int j0 = a.zv[z], U = a.zv[z + 1] - j0;
        const int g0 = a.zg[z], G = a.zg[z + 1] - g0;
        if (zone_smem_need(k, U, G) <= one_cta_smem) continue;   // the one-CTA solver's
        const int e0 = a.seg[j0];
        // shares: rows split at group boundaries (CL nearly equal group
        // counts), vertex j in CTA j / Ucap; every CTA computes all
        // boundaries, so every CTA derives the same layout
        const int Ucap = (U + CL - 1) / CL;
        if (tid <= CL) {
            const int gc = (int)(((long long)G * tid) / CL);
            gb[tid] = gc;
            rb[tid] = tid == CL ? k : a.gst[g0 + gc] - s0;
            const int vc = min(U, tid * Ucap);
            vb[tid] = vc;
            eb[tid] = a.seg[j0 + vc] - e0;
        }
        __syncthreads();
        int Kc = 0, Ec = 0, Gc = 0;
        for (int c = 0; c < CL; ++c) {
            Kc = max(Kc, rb[c + 1] - rb[c]);
            Ec = max(Ec, eb[c + 1] - eb[c]);
            Gc = max(Gc, gb[c + 1] - gb[c]);
        }
        const ClLayout L = cl_layout(Kc, Ucap, Ec, Gc);
        const double bb = [&] {
            double t = 0.0;
            for (int q = tid; q < k; q += nt) {
                const double bv = a.b64[s0 + q];
                t += bv * bv;
            }
            return block_sum_uniform(t, bredd);
        }();
        if (L.bytes > CL_SMEM) {
            // too large for the cluster's shared memory: the first CTA solves
            // it on global memory (the one-CTA path), the others go on
            if (rank == 0) solve_zone<CtaGroup, 0>(a, z, base, 0, bred, bredd, gs);
            continue;
        }
        const int r0 = rb[rank], kr = rb[rank + 1] - r0;            // own rows
        const int v0 = vb[rank], ur = vb[rank + 1] - v0;            // own vertices
        const int gg0 = gb[rank], gr = gb[rank + 1] - gg0;          // own groups
        const int ee0 = eb[rank], er = eb[rank + 1] - ee0;          // own CSR entries
        float4 *n4 = (float4 *)(base + L.o_n4);
        float4 *pinv = (float4 *)(base + L.o_pinv);
        int4 *vidx = (int4 *)(base + L.o_vidx);
        float4 *u = (float4 *)(base + L.o_u);
        float *f = (float *)(base + L.o_f);
        float *r = f, *p = f + Kc, *x = f + 2 * Kc, *sv = f + 3 * Kc, *w = f + 4 * Kc, *zz = f + 5 * Kc;
        float *winv = (float *)(base + L.o_winv);
        int *seg = (int *)(base + L.o_seg);
        int *ent = (int *)(base + L.o_ent);
        int *gst = (int *)(base + L.o_gst);
        // stage the own share
        for (int t = tid; t < kr; t += nt) {
            const int4 g = a.vidx[s0 + r0 + t];
            vidx[t] = make_int4(g.x - j0, g.y - j0, g.z - j0, g.w - j0);
            n4[t] = a.n32[s0 + r0 + t];
            pinv[t] = a.pinv[s0 + r0 + t];
            a.lam[s0 + r0 + t] = 0.0;
        }
        for (int q = tid; q <= gr; q += nt) gst[q] = a.gst[g0 + gg0 + q] - s0 - r0;
        for (int j = tid; j <= ur; j += nt) seg[j] = a.seg[j0 + v0 + j] - e0 - ee0;
        for (int j = tid; j < ur; j += nt) winv[j] = a.winv[j0 + v0 + j];
        for (int e = tid; e < er; e += nt) ent[e] = a.cval[e0 + ee0 + e] - 4 * s0;
        // the CTA that owns row s (rows split at rb)
        auto row_owner = [&](int sl) {
            int c = 0;
#pragma unroll
            for (int q = 1; q < CL; ++q) c += sl >= rb[q];
            return c;
        };
        const double target = a.rel_tol * a.rel_tol * bb;
        const float third = 1.0f / 3.0f;
        double rr = bb;
        int its = 0, rounds = 0;
        // the first round's right-hand side: b (lam = 0)
        for (int t = tid; t < kr; t += nt) r[t] = (float)a.b64[s0 + r0 + t];
        cl.sync();
        while (rr > target && rounds < a.max_refine) {
            for (int t = tid; t < kr; t += nt) { p[t] = 0.f; sv[t] = 0.f; x[t] = 0.f; }
            // ---- float32 PCG (Chronopoulos-Gear) on the float32 normals ----
            auto precond = [&]() {
                for (int g = tid; g < gr; g += nt) {
                    const int lo = gst[g], hi = gst[g + 1];
                    float rq[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) rq[q] = lo + q < hi ? r[lo + q] : 0.f;
                    for (int t = lo; t < hi; ++t) {
                        const float4 m = pinv[t];
                        zz[t] = m.x * rq[0] + m.y * rq[1] + m.z * rq[2] + m.w * rq[3];
                    }
                }
            };
            auto matvec_vertex = [&]() {   // u = M^-1 J^T z over the own vertices
                for (int j = tid; j < ur; j += nt) {
                    float a0 = 0.f, a1 = 0.f, a2 = 0.f;
                    for (int e = seg[j]; e < seg[j + 1]; ++e) {
                        const int c = ent[e];
                        const int sl = c >> 2;
                        const int ow = row_owner(sl);
                        const int li = sl - rb[ow];
                        const float zs = *cl.map_shared_rank(zz + li, ow);
                        const float4 nn = *cl.map_shared_rank(n4 + li, ow);
                        const float ps = ((c & 3) ? -third : 1.0f) * zs;
                        a0 += ps * nn.x;
                        a1 += ps * nn.y;
                        a2 += ps * nn.z;
                    }
                    const float wv = winv[j];
                    u[j] = make_float4(wv * a0, wv * a1, wv * a2, 0.f);
                }
            };
            auto matvec_rows = [&](float *ga, float *de, float *rh) {   // w = J u, partial sums
                for (int t = tid; t < kr; t += nt) {
                    const int4 g = vidx[t];
                    const float4 u0 = *cl.map_shared_rank(u + g.x % Ucap, g.x / Ucap);
                    const float4 u1 = *cl.map_shared_rank(u + g.y % Ucap, g.y / Ucap);
                    const float4 u2 = *cl.map_shared_rank(u + g.z % Ucap, g.z / Ucap);
                    const float4 u3 = *cl.map_shared_rank(u + g.w % Ucap, g.w / Ucap);
                    const float4 nn = n4[t];
                    const float ws = nn.x * (u0.x - (u1.x + u2.x + u3.x) * third) +
                                     nn.y * (u0.y - (u1.y + u2.y + u3.y) * third) +
                                     nn.z * (u0.z - (u1.z + u2.z + u3.z) * third);
                    w[t] = ws;
                    *ga += r[t] * zz[t];
                    *de += ws * zz[t];
                    *rh += r[t] * r[t];
                }
            };
            precond();
            cl.sync();
            matvec_vertex();
            cl.sync();
            float ga = 0.f, de = 0.f, rh = 0.f;
            matvec_rows(&ga, &de, &rh);
            float part[3], sums[3];
            cl_block3(ga, de, rh, bred, part);
            cl_reduce<float, 3>(cl, part, redf, sums);
            float gamma = sums[0], delta = sums[1], rho = sums[2];
            const float stop = (float)a.tol * (float)a.tol * rho;
            float alpha = gamma / delta, beta = 0.f;
            int it = 0;
            while (it < a.maxit && rho > stop && rho > 0.f && alpha > 0.f && isfinite(alpha)) {
                for (int g = tid; g < gr; g += nt) {
                    const int lo = gst[g], hi = gst[g + 1];
                    for (int t = lo; t < hi; ++t) {
                        const float ps = zz[t] + beta * p[t];
                        const float ss = w[t] + beta * sv[t];
                        p[t] = ps;
                        sv[t] = ss;
                        x[t] += alpha * ps;
                        r[t] -= alpha * ss;
                    }
                }
                __syncthreads();
                precond();
                cl.sync();
                matvec_vertex();
                cl.sync();
                ga = de = rh = 0.f;
                matvec_rows(&ga, &de, &rh);
                cl_block3(ga, de, rh, bred, part);
                cl_reduce<float, 3>(cl, part, redf, sums);
                beta = sums[0] / gamma;
                alpha = sums[0] / (sums[1] - beta * sums[0] / alpha);
                gamma = sums[0];
                rho = sums[2];
                ++it;
            }
            its += it;
            // ---- lam += x, then the zone's float64 residual b - A lam ----
            for (int t = tid; t < kr; t += nt) a.lam[s0 + r0 + t] += (double)x[t];
            __threadfence();
            cl.sync();
            const double third64 = 1.0 / 3.0;
            for (int j = tid; j < ur; j += nt) {
                double a0 = 0.0, a1 = 0.0, a2 = 0.0;
                for (int e = seg[j]; e < seg[j + 1]; ++e) {
                    const int c = ent[e];
                    const int sl = c >> 2;
                    const double ps = ((c & 3) ? -third64 : 1.0) * __ldcg(a.lam + s0 + sl);
                    const double4_32a nn = a.n64[s0 + sl];
                    a0 += ps * nn.x;
                    a1 += ps * nn.y;
                    a2 += ps * nn.z;
                }
                const double wv = (double)winv[j];
                double *uo = a.u64 + 3 * (size_t)(j0 + v0 + j);
                uo[0] = wv * a0;
                uo[1] = wv * a1;
                uo[2] = wv * a2;
            }
            __threadfence();
            cl.sync();
            double rrl = 0.0;
            for (int t = tid; t < kr; t += nt) {
                const int4 g = vidx[t];
                const double *ux = a.u64 + 3 * (size_t)(j0 + g.x), *ua = a.u64 + 3 * (size_t)(j0 + g.y);
                const double *ub = a.u64 + 3 * (size_t)(j0 + g.z), *uc = a.u64 + 3 * (size_t)(j0 + g.w);
                double d[3];
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    d[c] = __ldcg(ux + c) - (__ldcg(ua + c) + __ldcg(ub + c) + __ldcg(uc + c)) * third64;
                const double4_32a nn = a.n64[s0 + r0 + t];
                const double rv = a.b64[s0 + r0 + t] - (nn.x * d[0] + nn.y * d[1] + nn.z * d[2]);
                r[t] = (float)rv;
                rrl += rv * rv;
            }
            double pd[2] = {block_sum_uniform(rrl, bredd), 0.0}, sd[2];
            cl_reduce<double, 2>(cl, pd, redd, sd);
            rr = sd[0];
            ++rounds;
        }
        if (rank == 0 && tid == 0) {
            zone_finish(a, z, rr, bb, its, rounds, true);
            atomicAdd(&a.ctl[5], k);
            atomicAdd(&a.ctl[6], U);
        }
        // the shares (shared memory) of this zone are read by other CTAs until
        // every CTA has passed this barrier
        cl.sync();
    }
    cl.sync();
}

// |r| / |b| of the whole system from the zones' |r|^2 and |b|^2 (fixed
// summation order) to dres[0], |b|^2 to dres[1]; ctl[0] = converged
__global__ void __launch_bounds__(256) k_zone_final(const int *d_nz, const double *zres,
                                                    const double *zbb, double rel_tol,
                                                    double *dres, int *ctl) {
    HFCR_PDL_WAIT();
    __shared__ double redd[8];
    const int nz = *d_nz;
    double R = 0.0, Bn = 0.0;
    for (int z = threadIdx.x; z < nz; z += blockDim.x) {
        R += zres[z];
        Bn += zbb[z];
    }
    R = block_sum_uniform(R, redd);
    Bn = block_sum_uniform(Bn, redd);
    if (threadIdx.x == 0) {
        const double rel = Bn > 0.0 ? sqrt(R / Bn) : (R > 0.0 ? INFINITY : 0.0);
        dres[0] = rel;
        dres[1] = Bn;
        ctl[0] = rel <= rel_tol;
    }
}

// float64 residual, vertex half: u = M^-1 J^T lam
__global__ void k_res_vertex(const int *d_U, const int *seg, const int *cval, const float *winv,
                             const double4_32a *n64, const double *lam, double *u, const int *ctl) {
    HFCR_PDL_WAIT();
    if (ctl[0]) return;
    const int U = *d_U;
    const double third = 1.0 / 3.0;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < U; j += gridDim.x * blockDim.x) {
        double a0 = 0, a1 = 0, a2 = 0;
        for (int e = seg[j]; e < seg[j + 1]; ++e) {
            int v = cval[e];
            int s = v >> 2;
            double ps = ((v & 3) ? -third : 1.0) * lam[s];
            double4_32a n = n64[s];
            a0 += ps * n.x;
            a1 += ps * n.y;
            a2 += ps * n.z;
        }
        double w = (double)winv[j];
        u[3 * j] = w * a0;
        u[3 * j + 1] = w * a1;
        u[3 * j + 2] = w * a2;
    }
}

// float64 residual, stencil half: r = b - J u; per-block partial sums of
// r^2 and b^2 to red[blk] and red[RES_BLOCKS + blk].  The last block to
// finish (ticket counter) adds the partials in block order, records
// |r| / |b| in dres[0] and |b|^2 in dres[1], and sets ctl[0] when the
// relative residual meets rel_tol.
__global__ void k_res_stencil(const int *d_k, const int4 *vidx, const double4_32a *n64,
                              const double *b, const double *u, double *r, double *red,
                              int *ctl, unsigned *ticket, double rel_tol, double *dres,
                              int count_round) {
    HFCR_PDL_WAIT();
    __shared__ double sh[33];
    __shared__ bool last;
    if (ctl[0]) return;
    const int k = *d_k;
    const double third = 1.0 / 3.0;
    double rr = 0, bb = 0;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < k; s += gridDim.x * blockDim.x) {
        int4 vi = vidx[s];
        double4_32a n = n64[s];
        double d0 = u[3 * vi.x] - (u[3 * vi.y] + u[3 * vi.z] + u[3 * vi.w]) * third;
        double d1 = u[3 * vi.x + 1] - (u[3 * vi.y + 1] + u[3 * vi.z + 1] + u[3 * vi.w + 1]) * third;
        double d2 = u[3 * vi.x + 2] - (u[3 * vi.y + 2] + u[3 * vi.z + 2] + u[3 * vi.w + 2]) * third;
        double rs = b[s] - (n.x * d0 + n.y * d1 + n.z * d2);
        r[s] = rs;
        rr += rs * rs;
        bb += b[s] * b[s];
    }
    rr = block_sum(rr, sh);
    bb = block_sum(bb, sh);
    if (threadIdx.x == 0) {
        red[blockIdx.x] = rr;
        red[RES_BLOCKS + blockIdx.x] = bb;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last || threadIdx.x != 0) return;
    __threadfence();
    double R = 0, Bn = 0;
    for (int i = 0; i < (int)gridDim.x; ++i) {
        R += __ldcg(red + i);
        Bn += __ldcg(red + RES_BLOCKS + i);
    }
    double rel = Bn > 0 ? sqrt(R / Bn) : 0.0;
    dres[0] = rel;
    dres[1] = Bn;
    if (rel <= rel_tol) ctl[0] = 1;
    if (count_round) ctl[3] += 1;
    *ticket = 0;
}

__global__ void k_init_lam(const int *d_k, const double *b, double *lam, double *r) {
    HFCR_PDL_WAIT();
    const int k = *d_k;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < k; s += gridDim.x * blockDim.x) {
        lam[s] = 0.0;
        r[s] = b[s];
    }
}

// displacement of the touched vertices: dx = -M^-1 J^T lam (float64).
// apply 1: added to the positions; 0: written to the caller's arrays (mesh
// dtype); 2: written to the float64 field dA0 (x, y, z per global vertex)
__global__ void k_displace(const int *d_U, const int *seg, const int *cval, const float *winv,
                           const double4_32a *n64, const double *lam, const int *gvert, hfcr_mesh A,
                           hfcr_mesh B, int apply, void *dA0, void *dA1, void *dA2, void *dB0,
                           void *dB1, void *dB2, unsigned long long *max_dx) {
    HFCR_PDL_WAIT();
    const int U = *d_U;
    const double third = 1.0 / 3.0;
    double biggest = 0.0;  // the largest displacement component of this thread's vertices
    const int j_end = (U + (int)(gridDim.x * blockDim.x) - 1) / (int)(gridDim.x * blockDim.x) *
                      (int)(gridDim.x * blockDim.x);  // every thread of a warp runs the same trips
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < j_end; j += gridDim.x * blockDim.x) {
        if (j >= U) continue;
        double a0 = 0, a1 = 0, a2 = 0;
        for (int e = seg[j]; e < seg[j + 1]; ++e) {
            int v = cval[e];
            int s = v >> 2;
            double ps = ((v & 3) ? -third : 1.0) * lam[s];
            double4_32a n = n64[s];
            a0 += ps * n.x;
            a1 += ps * n.y;
            a2 += ps * n.z;
        }
        double w = (double)winv[j];
        double dx[3] = {-w * a0, -w * a1, -w * a2};
        biggest = fmax(biggest, fmax(fabs(dx[0]), fmax(fabs(dx[1]), fabs(dx[2]))));
        int g = gvert[j];
        if (apply == 2) {  // into the float64 field of the diffusion (AoS, global ids)
            double *f = (double *)dA0 + 3 * (size_t)g;
            f[0] = dx[0];
            f[1] = dx[1];
            f[2] = dx[2];
            continue;
        }
        const bool inA = g < A.n_verts;
        const hfcr_mesh &m = inA ? A : B;
        int lv = inA ? g : g - A.n_verts;
        if (apply) {
            void *P[3] = {m.x, m.y, m.z};
            for (int c = 0; c < 3; ++c) {
                if (m.dtype == HFCR_F32) {
                    float *pp = (float *)P[c] + lv;
                    *pp = (float)((double)*pp + dx[c]);
                } else {
                    double *pp = (double *)P[c] + lv;
                    *pp = *pp + dx[c];
                }
            }
        } else {
            void *O[3] = {inA ? dA0 : dB0, inA ? dA1 : dB1, inA ? dA2 : dB2};
            for (int c = 0; c < 3; ++c) {
                if (m.dtype == HFCR_F32) ((float *)O[c])[lv] = (float)dx[c];
                else ((double *)O[c])[lv] = dx[c];
            }
        }
    }
    warp_max_to(biggest, max_dx);
}

// ---------------------------------------------------------------------------
// The response setup in one cooperative launch: vertex CSR of the stencil
// entries, impact zones, zone-ordered rows, zone-ordered CSR, the groups of
// rows sharing x0 and the inverses of their blocks.  It computes exactly
// what the multi-kernel sequence of build_vertex_csr computes (the same
// stable sorts, the same union-find roots, hence the same arrays), in one
// launch instead of about twenty-five.  Up to SETUP_CTA_K stencils k_setup_cta
// has built the arrays and only the rows are left (setup_rows).  The
// elementwise phases run on every CTA taking part, separated by bounded
// grid-wide barriers, and data written by another CTA is read through L2.  Up
// to SETUP_SMALL_K stencils few CTAs take part (one per 1,024 entries) and the
// first CTA alone runs the sorts, the union-find (in shared memory) and the
// scans between two barriers; above, every CTA takes part in those too (the
// multi-CTA sort, union-find in global memory, the two-level scan).
// ---------------------------------------------------------------------------
constexpr int SETUP_SMALL_K = 8192;  // 4k <= SMALL_N sort keys, 32 KB of parents
constexpr int SETUP_SCAN_CHUNK = 4096;
constexpr int SETUP_ENTRIES_PER_CTA = 1024;

struct SetupArgs {
    const int *d_k;
    int cap, vbits, nA;
    const float *wA, *wB;
    const int4 *ids_raw;
    const double4_32a *n64_raw;
    const float4 *n32_raw;
    const double *b_raw;
    unsigned *ckey, *ckey_alt, *cflag;
    int *cval, *cval_alt;
    unsigned *zlab, *zlab_alt;
    int *zsrc, *zsrc_alt;
    unsigned *k2, *k2_alt;
    int *v2, *v2_alt;
    int *parent;  // union-find forest above SETUP_SMALL_K, then the position of each stencil
    int4 *ids;
    double4_32a *n64;
    float4 *n32;
    double *b;
    int *szone, *zs, *zv, *gst, *zg, *seg, *gvert;
    int4 *vidx;
    float *winv;
    float4 *pinv;
    int *d_n4, *d_U, *d_nz, *d_ng;
    unsigned *hist, *tot, *bar;
    uint32_t *status;
    int indexed;  // k_setup_cta ran before: up to SETUP_CTA_K stencils only the rows are left
};

// the CTAs taking part (blockIdx.x < parts) and their barrier
struct SetupSync {
    unsigned *bar;
    unsigned epoch;
    uint32_t *status;
    unsigned parts;
    __device__ bool sync() {
        if (parts == 1) {
            __syncthreads();
            return true;
        }
        return grid_barrier(bar, ++epoch, status, parts);
    }
};

__device__ __forceinline__ unsigned cta_sum_u(unsigned v) {
    __shared__ unsigned ws[TPB / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();  // ws is free of its previous use
    if (lane == 0) ws[w] = v;
    __syncthreads();
    unsigned t = 0;
#pragma unroll
    for (int q = 0; q < TPB / 32; ++q) t += ws[q];
    return t;
}

// exclusive scan of a[0..m) in place, the sum to *d_total; on return the
// scanned values and the sum are visible to every CTA taking part.  Small:
// the first CTA scans alone.  Otherwise chunks of SETUP_SCAN_CHUNK: chunk
// sums, a barrier, each chunk scanned from the sum of the chunks before it.
__device__ __forceinline__ bool setup_scan(SetupSync &g, bool small, unsigned *a, int m,
                                           unsigned *part, int *d_total, unsigned &total) {
    if (small) {
        if (blockIdx.x == 0) {
            const unsigned t = block_scan_excl<TPB, true>(a, m);
            if (threadIdx.x == 0) *d_total = (int)t;
        }
        if (!g.sync()) return false;
        total = (unsigned)__ldcg(d_total);
        return true;
    }
    const int nc = (m + SETUP_SCAN_CHUNK - 1) / SETUP_SCAN_CHUNK;
    for (int c = blockIdx.x; c < nc; c += g.parts) {
        const int base = c * SETUP_SCAN_CHUNK, end = min(m, base + SETUP_SCAN_CHUNK);
        unsigned x = 0;
        for (int i = base + threadIdx.x; i < end; i += TPB) x += __ldcg(a + i);
        x = cta_sum_u(x);
        if (threadIdx.x == 0) part[c] = x;
    }
    if (!g.sync()) return false;
    for (int c = blockIdx.x; c < nc; c += g.parts) {
        unsigned x = 0;
        for (int i = threadIdx.x; i < c; i += TPB) x += __ldcg(part + i);
        const unsigned off = cta_sum_u(x);
        const int base = c * SETUP_SCAN_CHUNK;
        block_scan_excl<TPB, true>(a + base, min(m - base, SETUP_SCAN_CHUNK), off);
    }
    unsigned x = 0;
    for (int i = threadIdx.x; i < nc; i += TPB) x += __ldcg(part + i);
    total = cta_sum_u(x);
    if (blockIdx.x == 0 && threadIdx.x == 0) *d_total = (int)total;
    return g.sync();
}

// stable sort of (key, val) pairs over `bits` bits (a multiple of 8); the
// result is in (k1, v1) after an odd number of passes.  One CTA taking
// part: the single-CTA sort; otherwise every CTA taking part (at most one
// tile each on small inputs: no scan phase).
__device__ __forceinline__ bool setup_sort(SetupSync &g, bool small, unsigned *k0, int *v0,
                                           unsigned *k1, int *v1, int n, int bits,
                                           const SetupArgs &a, SortSmem &sm) {
    if (small && g.parts == 1) {
        sort_small_body<unsigned, true, true>(k0, v0, k1, v1, n, bits, sm);
        return g.sync();
    }
    return sort_grid_body<unsigned, true>(k0, v0, k1, v1, n, bits, a.hist, a.tot, g.bar, g.epoch,
                                          g.status, sm, g.parts);
}

__device__ __forceinline__ int setup_bits(int n) {  // 8 x the passes for keys < n (n >= 1)
    int b = 1;
    while ((1 << b) < n) ++b;
    return 8 * ((b + 7) / 8);
}

__device__ __forceinline__ bool group_start_l2(const int4 *ids, const int *szone, const int *zs,
                                               int t) {
    const int zs0 = __ldcg(zs + __ldcg(szone + t)), x0 = __ldcg(&ids[t].x);
    int rs = t;
    while (rs > zs0 && __ldcg(&ids[rs - 1].x) == x0) --rs;
    return ((t - rs) % GMAX) == 0;
}

// unites the zones of stencils s0 and s1 (the smaller root becomes the
// root); SH: parents in shared memory
template <bool SH>
__device__ __forceinline__ void setup_unite(int *par, int s0, int s1, uint32_t *status) {
    int a = s0, b = s1, guard = 0;
    while (true) {
        if constexpr (SH) {
            a = uf_find_s(par, a);
            b = uf_find_s(par, b);
        } else {
            a = uf_find(par, a);
            b = uf_find(par, b);
        }
        if (a == b) break;
        if (a < b) { int t = a; a = b; b = t; }
        const int old = atomicCAS(par + a, a, b);
        if (old == a) break;
        a = old;
        if (++guard > (1 << 24)) { atomicOr(status, ST_TIMEOUT); break; }
    }
}

// Impact zones of up to SETUP_SMALL_K stencils by one CTA, in shared
// memory: connected components of the stencils, two stencils being
// adjacent when consecutive entries of the vertex-sorted list (ck1, cv1)
// share a vertex.  Min-label hooking with shortcutting (the FastSV scheme of
// Zhang, Azad and Hu, 2020): every sweep hooks the parent of each end of an
// edge, and each end itself, under the smaller of their grandparents
// (atomicMin), then every stencil jumps to its grandparent; labels only
// fall and stay inside their component, so at the first sweep that changes
// nothing every stencil points straight at the smallest stencil of its
// zone (the root the lock-free union-find gives too).  After SV_SWEEPS
// sweeps without convergence the forest (every parent smaller than its
// child, inside the same zone) is finished by the union-find.
constexpr int SV_SWEEPS = 64;

// edge[i] (i < n4): the stencils (u << 16 | v) of entries i and i - 1 of the
// vertex-sorted list when they share a vertex, NO_EDGE otherwise
constexpr unsigned NO_EDGE = 0xffffffffu;

__device__ void zones_min_label(int *f, int k, const unsigned *edge, int n4, uint32_t *status) {
    __shared__ int changed;
    for (int s = threadIdx.x; s < k; s += TPB) f[s] = s;
    if (threadIdx.x == 0) changed = 0;
    __syncthreads();
    int again = 1;
    for (int sweep = 0; sweep < SV_SWEEPS; ++sweep) {
        bool ch = false;
        for (int i = threadIdx.x + 1; i < n4; i += TPB) {
            const unsigned e = edge[i];
            if (e == NO_EDGE) continue;
            const int u = (int)(e >> 16), v = (int)(e & 0xffffu);
            const int fu = f[u], fv = f[v];
            const int m = min(f[fu], f[fv]);
            ch |= atomicMin(f + fu, m) > m;
            ch |= atomicMin(f + fv, m) > m;
            ch |= atomicMin(f + u, m) > m;
            ch |= atomicMin(f + v, m) > m;
        }
        __syncthreads();
        for (int s = threadIdx.x; s < k; s += TPB) {
            const int gp = f[f[s]];
            ch |= atomicMin(f + s, gp) > gp;
        }
        if (ch) changed = 1;
        __syncthreads();
        again = changed;
        __syncthreads();
        if (!again) break;
        if (threadIdx.x == 0) changed = 0;  // written again only after the next sweep's barrier
    }
    if (again) {
        for (int i = threadIdx.x + 1; i < n4; i += TPB) {
            const unsigned e = edge[i];
            if (e != NO_EDGE) setup_unite<true>(f, (int)(e >> 16), (int)(e & 0xffffu), status);
        }
        __syncthreads();
    }
}

// word of the barrier row raised when the groups are built (zeroed with
// the barrier counter before the launch)
constexpr int SETUP_READY = 1;

// the inverse blocks of CTAs first .. first + n - 1 (consecutive groups on
// different CTAs)
__device__ __forceinline__ void setup_inverses(const SetupArgs &a, int first, int n) {
    group_inverses<L2Ld>(0, (int)(threadIdx.x >> 5) * n + (int)blockIdx.x - first, n * (TPB / 32), __ldcg(a.d_ng),
                         a.gst, a.ids, a.n64, a.nA, a.wA, a.wB, a.pinv);
}

// a CTA not taking part in the phases (first = the first such CTA): waits
// (bounded, like the barrier) for the groups, then computes its share of
// the inverse blocks
__device__ void setup_helper(const SetupArgs &a, int first) {
    __shared__ int go;
    if (threadIdx.x == 0) {
        go = 0;
        long long spins = 0;
        while (true) {
            unsigned seen;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen)
                         : "l"(a.bar + SETUP_READY) : "memory");
            if (seen) { go = 1; break; }
            if (*(volatile uint32_t *)a.status & ST_TIMEOUT) break;
            if (++spins > BARRIER_SPIN_LIMIT) {
                atomicOr(a.status, ST_TIMEOUT);
                break;
            }
            __nanosleep(100);
        }
    }
    __syncthreads();
    if (go) setup_inverses(a, first, (int)gridDim.x - first);
}

__device__ bool setup_phases(SetupSync &g, const SetupArgs &a, int k, SortSmem &sm, int *par_s) {
    const bool small = k <= SETUP_SMALL_K;
    const int tid = blockIdx.x * TPB + threadIdx.x, nt = (int)g.parts * TPB, n4 = 4 * k;
    if (tid == 0) *a.d_n4 = n4;
    if (k == 0) {
        if (tid == 0) { *a.d_U = 0; *a.d_nz = 0; *a.d_ng = 0; }
        return true;
    }
    // vertex CSR: entries (vertex, 4 s + role) sorted by vertex
    for (int i = tid; i < n4; i += nt) {
        a.ckey[i] = (unsigned)((const int *)a.ids_raw)[i];
        a.cval[i] = i;
    }
    if (!g.sync()) return false;
    const bool f1 = (a.vbits / 8) & 1;
    const unsigned *ck1 = f1 ? a.ckey_alt : a.ckey;
    const int *cv1 = f1 ? a.cval_alt : a.cval;
    // impact zones: stencils of consecutive entries on the same vertex are
    // united; every zone's root is its smallest stencil.  Then the rows
    // regrouped zone by zone (zones in the order of their root).
    const int zbits = setup_bits(k);
    const bool f2 = (zbits / 8) & 1;
    const unsigned *zl = f2 ? a.zlab_alt : a.zlab;
    const int *zr = f2 ? a.zsrc_alt : a.zsrc;
    if (small) {
        // the entries sorted by every CTA taking part (one CTA: by itself),
        // then the zones, the labels and their sort in the first CTA
        if (g.parts > 1 &&
            !sort_grid_body<unsigned, true>(a.ckey, a.cval, a.ckey_alt, a.cval_alt, n4, a.vbits,
                                            a.hist, a.tot, g.bar, g.epoch, g.status, sm, g.parts))
            return false;
        if (blockIdx.x == 0) {
            if (g.parts == 1)
                sort_small_body<unsigned, true, true>(a.ckey, a.cval, a.ckey_alt, a.cval_alt, n4,
                                                      a.vbits, sm);
            int *par = par_s;  // overlays the sort's shared memory (the sort is done)
            // the adjacent pairs of sorted entries, read once through L2
            // (other CTAs wrote them; eight entries' loads in flight per
            // thread) and packed into cflag (free here)
            for (int i0 = 0; i0 < n4; i0 += 8 * TPB) {
                unsigned kc[8], kb[8];
                int vc[8], vb[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int i = i0 + q * TPB + threadIdx.x;
                    const bool ok = i > 0 && i < n4;
                    kc[q] = ok ? __ldcg(ck1 + i) : 0u;
                    kb[q] = ok ? __ldcg(ck1 + i - 1) : 1u;
                    vc[q] = ok ? __ldcg(cv1 + i) : 0;
                    vb[q] = ok ? __ldcg(cv1 + i - 1) : 0;
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int i = i0 + q * TPB + threadIdx.x;
                    if (i < n4)
                        a.cflag[i] = kc[q] == kb[q]
                                         ? (unsigned)(vc[q] >> 2) << 16 | (unsigned)(vb[q] >> 2)
                                         : NO_EDGE;
                }
            }
            __syncthreads();
            zones_min_label(par, k, a.cflag, n4, a.status);
            for (int s = threadIdx.x; s < k; s += TPB) {
                a.zlab[s] = (unsigned)uf_find_s(par, s);
                a.zsrc[s] = s;
            }
            __syncthreads();
            sort_small_body<unsigned, true>(a.zlab, a.zsrc, a.zlab_alt, a.zsrc_alt, k, zbits, sm);
            for (int t = threadIdx.x; t < k; t += TPB)
                a.cflag[t] = (t == 0 || zl[t] != zl[t - 1]) ? 1u : 0u;
            __syncthreads();
        }
    } else {
        if (!setup_sort(g, false, a.ckey, a.cval, a.ckey_alt, a.cval_alt, n4, a.vbits, a, sm))
            return false;
        int *par = a.parent;
        for (int s = tid; s < k; s += nt) par[s] = s;
        if (!g.sync()) return false;
        for (int i = tid + 1; i < n4; i += nt)
            if (__ldcg(ck1 + i) == __ldcg(ck1 + i - 1))
                setup_unite<false>(par, __ldcg(cv1 + i) >> 2, __ldcg(cv1 + i - 1) >> 2, a.status);
        if (!g.sync()) return false;
        for (int s = tid; s < k; s += nt) {
            a.zlab[s] = (unsigned)uf_find(par, s);
            a.zsrc[s] = s;
        }
        if (!g.sync()) return false;
        if (!setup_sort(g, false, a.zlab, a.zsrc, a.zlab_alt, a.zsrc_alt, k, zbits, a, sm))
            return false;
        for (int t = tid; t < k; t += nt)
            a.cflag[t] = (t == 0 || __ldcg(zl + t) != __ldcg(zl + t - 1)) ? 1u : 0u;
        if (!g.sync()) return false;
    }
    unsigned nz;
    if (!setup_scan(g, small, a.cflag, k, a.hist, a.d_nz, nz)) return false;
    int *pos_of = a.parent;
    for (int t = tid; t < k; t += nt) {
        const int src = __ldcg(zr + t);
        const unsigned f = (t == 0 || __ldcg(zl + t) != __ldcg(zl + t - 1)) ? 1u : 0u;
        const int z = (int)(__ldcg(a.cflag + t) + f) - 1;
        a.szone[t] = z;
        pos_of[src] = t;
        if (f) a.zs[z] = t;
        if (t == k - 1) a.zs[z + 1] = k;
        a.ids[t] = a.ids_raw[src];
        a.n64[t] = a.n64_raw[src];
        a.n32[t] = a.n32_raw[src];
        a.b[t] = a.b_raw[src];
    }
    if (!g.sync()) return false;
    // groups of rows sharing x0 (at most GMAX rows each)
    for (int t = tid; t < k; t += nt)
        a.cflag[t] = group_start_l2(a.ids, a.szone, a.zs, t) ? 1u : 0u;
    if (!g.sync()) return false;
    unsigned ng;
    if (!setup_scan(g, small, a.cflag, k, a.hist, a.d_ng, ng)) return false;
    for (int t = tid; t < k; t += nt) {
        const bool st = group_start_l2(a.ids, a.szone, a.zs, t);
        const int gi = (int)__ldcg(a.cflag + t);
        if (st) {
            a.gst[gi] = t;
            const int z = __ldcg(a.szone + t);
            if (__ldcg(a.zs + z) == t) a.zg[z] = gi;
        }
        if (t == k - 1) {
            a.gst[ng] = k;
            a.zg[nz] = (int)ng;
        }
    }
    // the inverse blocks (float64) need only the groups, the zone-ordered
    // rows and the masses: the CTAs not taking part compute them while the
    // others build the zone-ordered CSR (they wait for this flag,
    // SETUP_READY); without such CTAs the others compute them at the end
    const bool helpers = g.parts < gridDim.x;
    if (helpers) {
        __threadfence();  // the groups are written before the flag below
        if (!g.sync()) return false;
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(a.bar + SETUP_READY, 1u);
    }
    // zone-ordered CSR: the vertex-ordered entries re-sorted stably by zone
    // (an odd pass count starts from the spare buffers, so that the sorted
    // entries end in v2, where the solver reads them)
    const int qbits = setup_bits((int)nz);
    const bool qodd = (qbits / 8) & 1;
    unsigned *k2in = qodd ? a.k2_alt : a.k2, *k2out = qodd ? a.k2 : a.k2_alt;
    int *v2in = qodd ? a.v2_alt : a.v2, *v2out = qodd ? a.v2 : a.v2_alt;
    for (int i = tid; i < n4; i += nt) {
        const int e = __ldcg(cv1 + i);
        const int t = __ldcg(pos_of + (e >> 2));
        k2in[i] = (unsigned)__ldcg(a.szone + t);
        v2in[i] = 4 * t + (e & 3);
    }
    if (!g.sync()) return false;
    if (!setup_sort(g, small, k2in, v2in, k2out, v2out, n4, qbits, a, sm)) return false;
    const unsigned *zk = a.k2;
    const int *val = a.v2;
    const int *idsi = (const int *)a.ids;
    for (int i = tid; i < n4; i += nt)
        a.cflag[i] = (i == 0 || __ldcg(idsi + __ldcg(val + i)) != __ldcg(idsi + __ldcg(val + i - 1)))
                         ? 1u : 0u;
    if (!g.sync()) return false;
    unsigned U;
    if (!setup_scan(g, small, a.cflag, n4, a.hist, a.d_U, U)) return false;
    for (int i = tid; i < n4; i += nt) {
        const int vi = __ldcg(val + i);
        const int gv = __ldcg(idsi + vi);
        const unsigned f = (i == 0 || gv != __ldcg(idsi + __ldcg(val + i - 1))) ? 1u : 0u;
        const int j = (int)(__ldcg(a.cflag + i) + f) - 1;
        ((int *)a.vidx)[vi] = j;
        if (f) {
            a.seg[j] = i;
            a.gvert[j] = gv;
            const float *w = gv < a.nA ? a.wA : a.wB;
            const int lv = gv < a.nA ? gv : gv - a.nA;
            a.winv[j] = w ? w[lv] : 1.0f;
            const unsigned zi = __ldcg(zk + i);
            if (i == 0 || zi != __ldcg(zk + i - 1)) a.zv[zi] = j;
        }
        if (i == n4 - 1) {
            a.seg[j + 1] = n4;
            a.zv[nz] = j + 1;
        }
    }
    if (!g.sync()) return false;
    if (!helpers) setup_inverses(a, 0, (int)g.parts);
    return true;
}

// ---------------------------------------------------------------------------
// The setup of up to SETUP_CTA_K stencils without a sort of the entries: one
// CTA of 1,024 threads builds every index array in shared memory, then the
// rows (gather and inverse blocks, all elementwise) go to a grid.
//   - A hash table of the touched vertices; each vertex's first entry (its
//     smallest 4 s + role) is its head, and a stencil and the heads of its
//     vertices are of one zone (sweeps of hooking roots; a zone's root is its
//     smallest stencil).
//   - Zones numbered by their roots (scan), rows placed by a stable counting
//     sort of the zone numbers (8 bits a pass, ranks by warp matches).
//   - Vertices numbered in the order of their heads among the placed rows,
//     which is zone by zone; one scan gives the number and the start of each
//     one's list, a cursor places the entries, and every list is sorted (each
//     entry counts the smaller ones; a warp, or, past SETUP_LONG entries, a
//     bitmap by the whole CTA), so the result does not depend on the order of
//     the atomics.
// The numbering of a zone's vertices differs from the sorted one of the other
// paths; every sum over a list or a zone's rows keeps its order, hence its
// bits.  Bound by the latency of about 25 barriers and shared-memory phases:
// 1,955 rows in 21 zones 186 -> 37 us, 107 rows 85 -> 12 us, 1,219 rows in one
// zone 100 -> 24 us, and 13 us more for the rows' grid, against the
// cooperative launch's sorts.
// ---------------------------------------------------------------------------
constexpr int SETUP_CTA_K = 4096;
constexpr int SETUP_CTA_THREADS = 1024;
constexpr int SETUP_ROWS = SETUP_CTA_K / SETUP_CTA_THREADS;  // rows of a thread at most
constexpr int SETUP_TAB = 21 * SETUP_CTA_K / 4;              // slots: 1.3 x the entries
constexpr int SETUP_SHORT = 16, SETUP_LONG = 128;            // list lengths
static_assert(SETUP_TAB <= 0x8000, "a slot and a flag fit 16 bits");
static_assert(4 * SETUP_CTA_K <= 0x8000, "entries fit 16 bits");

struct SetupCtaSmem {
    // a slot's vertex, then its head, then its list's length, then the vertex's
    // number and its list's cursor
    unsigned tab[SETUP_TAB];
    uint16_t slot[4 * SETUP_CTA_K];  // of each entry; bit 15: the entry is its vertex's head
    union {
        int par[SETUP_CTA_K];
        uint16_t hist[256 * 32];     // digit-major, one column per warp
        uint16_t cval[4 * SETUP_CTA_K];
    } u;
    uint16_t key[2][SETUP_CTA_K], src[2][SETUP_CTA_K];
    uint16_t pos[SETUP_CTA_K];
    uint16_t start[4 * SETUP_CTA_K + 2];  // of each vertex's list
    unsigned bits[4 * SETUP_CTA_K / 32];
    unsigned ws[2][32];
    int n_list;
};

// exclusive scan (sum, or maximum) over the CTA; flip alternates the two
// rows of ws, so that one barrier is enough
template <bool MAX>
__device__ __forceinline__ unsigned setup_cta_scan(unsigned v, unsigned (*ws)[32], int &flip, unsigned &total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto op = [](unsigned a, unsigned b) { return MAX ? max(a, b) : a + b; };
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x = op(x, y);
    }
    if (lane == 31) ws[flip][w] = x;
    __syncthreads();
    unsigned y = ws[flip][lane];
    flip ^= 1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= o) y = op(y, t);
    }
    total = __shfl_sync(0xffffffffu, y, 31);
    unsigned before = __shfl_sync(0xffffffffu, y, w ? w - 1 : 0);
    if (w == 0) before = 0;
    unsigned ex = __shfl_up_sync(0xffffffffu, x, 1);
    if (lane == 0) ex = 0;
    return op(before, ex);
}

__global__ void __launch_bounds__(SETUP_CTA_THREADS, 1) k_setup_cta(SetupArgs a) {
    HFCR_PDL_WAIT();
    extern __shared__ float4 smem4[];
    SetupCtaSmem &m = *(SetupCtaSmem *)smem4;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int k = max(0, min(*a.d_k, a.cap));
    if (tid < 2) a.bar[tid] = 0u;  // k_setup's barrier counter and ready flag
    if (k > SETUP_CTA_K) return;
    const int n4 = 4 * k;
    if (tid == 0) *a.d_n4 = n4;
    if (k == 0) {
        if (tid == 0) { *a.d_U = 0; *a.d_nz = 0; *a.d_ng = 0; }
        return;
    }
    // a thread's rows: per consecutive ones
    const int per = (k + SETUP_CTA_THREADS - 1) / SETUP_CTA_THREADS;
    const int r0 = tid * per, nr = max(0, min(per, k - r0));
    const unsigned T = 21u * (unsigned)k / 4u;
    int flip = 0;
    int4 q[SETUP_ROWS];
#pragma unroll
    for (int i = 0; i < SETUP_ROWS; ++i)
        q[i] = i < nr ? a.ids_raw[r0 + i] : make_int4(0, 0, 0, 0);
    for (int i = tid; i < (int)T; i += SETUP_CTA_THREADS) m.tab[i] = 0xffffffffu;
    __syncthreads();
    // the table (Fibonacci hashing, linear probing; reads first, since most
    // entries find their vertex there)
#pragma unroll
    for (int i = 0; i < SETUP_ROWS; ++i) {
        if (i >= nr) break;
        const unsigned v[4] = {(unsigned)q[i].x, (unsigned)q[i].y, (unsigned)q[i].z, (unsigned)q[i].w};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            unsigned h = __umulhi(v[r] * 0x9e3779b1u, T);
            while (true) {  // ends: there are more slots than entries
                unsigned old = *(volatile unsigned *)&m.tab[h];
                if (old == 0xffffffffu) old = atomicCAS(&m.tab[h], 0xffffffffu, v[r]);
                if (old == 0xffffffffu || old == v[r]) break;
                if (++h == T) h = 0;
            }
            m.slot[4 * (r0 + i) + r] = (uint16_t)h;
        }
    }
    __syncthreads();
    for (int e = 4 * r0; e < 4 * (r0 + nr); ++e) m.tab[m.slot[e]] = 0xffffffffu;
    __syncthreads();
    for (int e = 4 * r0; e < 4 * (r0 + nr); ++e) atomicMin(&m.tab[m.slot[e]], (unsigned)e);
    __syncthreads();
    // a stencil's first parent: the smallest of its vertices' heads.  Then
    // sweeps: every tree hooks the roots its stencils' vertices reach under
    // the smallest of them, until no vertex joins two trees (parents are
    // smaller than children, so a zone's root is its smallest stencil)
    uint16_t *snap = m.start;  // the roots of a sweep
    unsigned hd[SETUP_ROWS][2];
#pragma unroll
    for (int i = 0; i < SETUP_ROWS; ++i) {
        if (i >= nr) break;
        unsigned lo = r0 + i, h[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int e = 4 * (r0 + i) + r;
            const unsigned sl = m.slot[e];
            h[r] = m.tab[sl];
            if ((int)h[r] == e) m.slot[e] = (uint16_t)(sl | 0x8000u);
            h[r] >>= 2;
            lo = min(lo, h[r]);
        }
        m.u.par[r0 + i] = (int)lo;
        hd[i][0] = h[0] | h[1] << 16;
        hd[i][1] = h[2] | h[3] << 16;
    }
    __syncthreads();
    while (true) {
#pragma unroll
        for (int i = 0; i < SETUP_ROWS; ++i)
            if (i < nr) snap[r0 + i] = (uint16_t)uf_find_s((volatile int *)m.u.par, r0 + i);
        __syncthreads();
        bool hooked = false;
#pragma unroll
        for (int i = 0; i < SETUP_ROWS; ++i) {
            if (i >= nr) break;
            const int x[5] = {snap[r0 + i], snap[hd[i][0] & 0xffffu], snap[hd[i][0] >> 16],
                              snap[hd[i][1] & 0xffffu], snap[hd[i][1] >> 16]};
            const int lo = min(min(min(x[0], x[1]), min(x[2], x[3])), x[4]);
#pragma unroll
            for (int r = 0; r < 5; ++r)
                if (x[r] > lo) {
                    atomicMin(&m.u.par[x[r]], lo);
                    hooked = true;
                }
        }
        if (!__syncthreads_or(hooked)) break;
    }
    // zones in the order of their roots; the list lengths start at 0
    int root[SETUP_ROWS];
    unsigned cnt = 0;
#pragma unroll
    for (int i = 0; i < SETUP_ROWS; ++i) {
        root[i] = -1;
        if (i >= nr) continue;
        root[i] = snap[r0 + i];
        cnt += root[i] == r0 + i;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const unsigned sl = m.slot[4 * (r0 + i) + r];
            if (sl & 0x8000u) m.tab[sl & 0x7fffu] = 0u;
        }
    }
    unsigned nz;
    unsigned zi = setup_cta_scan<false>(cnt, m.ws, flip, nz);
#pragma unroll
    for (int i = 0; i < SETUP_ROWS; ++i)
        if (root[i] >= 0 && root[i] == r0 + i) m.pos[r0 + i] = (uint16_t)zi++;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SETUP_ROWS; ++i) {
        if (i >= nr) break;
        m.key[0][r0 + i] = m.pos[root[i]];
        m.src[0][r0 + i] = (uint16_t)(r0 + i);
    }
    // the list lengths
    for (int e = 4 * r0; e < 4 * (r0 + nr); ++e) atomicAdd(&m.tab[m.slot[e] & 0x7fffu], 1u);
    int f = 0;
    for (int shift = 0; (int)nz - 1 >> shift; shift += 8) {
        __syncthreads();  // the keys; par and the previous counts are no longer read
        for (int i = tid; i < 256 * 32 / 2; i += SETUP_CTA_THREADS) ((unsigned *)m.u.hist)[i] = 0u;
        __syncthreads();
        // rows 32 per * w + 32 i + lane of warp w
        unsigned dig[SETUP_ROWS], rank[SETUP_ROWS];
#pragma unroll
        for (int i = 0; i < SETUP_ROWS; ++i) {
            if (i >= per) break;
            const int t = 32 * (per * w + i) + lane;
            dig[i] = t < k ? (m.key[f][t] >> shift) & 255u : 256u;
            const unsigned same = __match_any_sync(0xffffffffu, dig[i]);
            const unsigned before = dig[i] < 256u ? m.u.hist[dig[i] * 32 + w] : 0u;
            rank[i] = before + __popc(same & ((1u << lane) - 1u));
            __syncwarp();
            if (dig[i] < 256u && lane == __ffs(same) - 1)
                m.u.hist[dig[i] * 32 + w] = (uint16_t)(before + __popc(same));
            __syncwarp();
        }
        __syncthreads();
        uint4 h = ((uint4 *)m.u.hist)[tid];
        unsigned hv[8] = {h.x & 0xffffu, h.x >> 16, h.y & 0xffffu, h.y >> 16,
                          h.z & 0xffffu, h.z >> 16, h.w & 0xffffu, h.w >> 16};
        unsigned sum = 0, all;
#pragma unroll
        for (int i = 0; i < 8; ++i) sum += hv[i];
        unsigned at = setup_cta_scan<false>(sum, m.ws, flip, all);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const unsigned c = hv[i];
            hv[i] = at;
            at += c;
        }
        ((uint4 *)m.u.hist)[tid] = make_uint4(hv[0] | hv[1] << 16, hv[2] | hv[3] << 16,
                                              hv[4] | hv[5] << 16, hv[6] | hv[7] << 16);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < SETUP_ROWS; ++i) {
            if (i >= per) break;
            const int t = 32 * (per * w + i) + lane;
            if (t >= k) continue;
            const unsigned d = m.u.hist[dig[i] * 32 + w] + rank[i];
            m.key[f ^ 1][d] = m.key[f][t];
            m.src[f ^ 1][d] = m.src[f][t];
        }
        f ^= 1;
    }
    __syncthreads();
    // rows: zone, source, the groups of rows sharing x0 (GMAX rows at most)
    const uint16_t *key = m.key[f], *src = m.src[f];
    unsigned last_run = 0, heads = 0;  // this thread's last run start + 1; its vertices and entries
    unsigned run[SETUP_ROWS];
#pragma unroll
    for (int i = 0; i < SETUP_ROWS; ++i) {
        if (i >= nr) break;
        const int t = r0 + i, sr = src[t], z = key[t];
        const bool first = t == 0 || key[t - 1] != z;
        const unsigned x0 = m.slot[4 * sr] & 0x7fffu;
        q[i] = a.ids_raw[sr];
        a.szone[t] = z;
        a.zsrc[t] = sr;
        if (first) a.zs[z] = t;
        if (first || (m.slot[4 * src[t - 1]] & 0x7fffu) != x0) last_run = (unsigned)t + 1u;
        run[i] = last_run;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const unsigned sl = m.slot[4 * sr + r];
            if (sl & 0x8000u) heads += 0x10000u + m.tab[sl & 0x7fffu];
        }
    }
    unsigned total;
    const unsigned run_before = setup_cta_scan<true>(last_run, m.ws, flip, total);
    cnt = 0;
#pragma unroll
    for (int i = 0; i < SETUP_ROWS; ++i) {
        if (i >= nr) break;
        const int t = r0 + i, rs = (int)(run[i] ? run[i] : run_before) - 1;
        run[i] = (t - rs) % GMAX == 0;
        cnt += run[i];
    }
    unsigned ng, Un;
    unsigned gi = setup_cta_scan<false>(cnt, m.ws, flip, ng);
    const unsigned base = setup_cta_scan<false>(heads, m.ws, flip, Un);
    const int U = (int)(Un >> 16);
    unsigned at = base;  // vertex number << 16 | list start
#pragma unroll
    for (int i = 0; i < SETUP_ROWS; ++i) {
        if (i >= nr) break;
        const int t = r0 + i, sr = src[t], z = key[t];
        const bool first = t == 0 || key[t - 1] != z;
        if (run[i]) {
            a.gst[gi] = t;
            if (first) a.zg[z] = (int)gi;
            ++gi;
        }
        if (first) a.zv[z] = (int)(at >> 16);  // a zone's first entry is a head
        const int v[4] = {q[i].x, q[i].y, q[i].z, q[i].w};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const unsigned sl = m.slot[4 * sr + r];
            if (!(sl & 0x8000u)) continue;
            const int j = (int)(at >> 16);
            const unsigned c = m.tab[sl & 0x7fffu];
            m.tab[sl & 0x7fffu] = at;
            a.seg[j] = (int)(at & 0xffffu);
            m.start[j] = (uint16_t)(at & 0xffffu);
            a.gvert[j] = v[r];
            const float *wm = v[r] < a.nA ? a.wA : a.wB;
            a.winv[j] = wm ? wm[v[r] < a.nA ? v[r] : v[r] - a.nA] : 1.0f;
            at += 0x10000u + c;
        }
    }
    if (tid == 0) {
        a.zs[nz] = k;
        a.gst[ng] = k;
        a.zg[nz] = (int)ng;
        a.seg[U] = n4;
        a.zv[nz] = U;
        *a.d_nz = (int)nz;
        *a.d_ng = (int)ng;
        *a.d_U = U;
        m.start[U] = (uint16_t)n4;
        m.n_list = 0;
    }
    __syncthreads();
    // the entries into their vertices' lists
#pragma unroll
    for (int i = 0; i < SETUP_ROWS; ++i) {
        if (i >= nr) break;
        const int t = r0 + i, sr = src[t];
        int j[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const unsigned o = atomicAdd(&m.tab[m.slot[4 * sr + r] & 0x7fffu], 1u);
            j[r] = (int)(o >> 16);
            m.u.cval[o & 0xffffu] = (uint16_t)(4 * t + r);
        }
        q[i] = make_int4(j[0], j[1], j[2], j[3]);
        a.vidx[t] = q[i];
    }
    __syncthreads();
    // each list ascending: a short list's entries find their own ranks, a
    // longer one is noted by its first entry to be placed
#pragma unroll
    for (int i = 0; i < SETUP_ROWS; ++i) {
        if (i >= nr) break;
        const int j[4] = {q[i].x, q[i].y, q[i].z, q[i].w};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int e = 4 * (r0 + i) + r, lo = m.start[j[r]], hi = m.start[j[r] + 1];
            if (hi - lo <= SETUP_SHORT) {
                int at = lo;
                for (int x = lo; x < hi; ++x) at += (int)m.u.cval[x] < e;
                a.v2[at] = e;
            } else if ((int)m.u.cval[lo] == e) {
                const int n = atomicAdd(&m.n_list, 1);  // at most 4 k / 17 lists
                m.pos[2 * n] = (uint16_t)lo;
                m.pos[2 * n + 1] = (uint16_t)hi;
            }
        }
    }
    __syncthreads();
    const int nl = m.n_list;
    for (int x = w; x < nl; x += 32) {
        const int b = m.pos[2 * x], n = m.pos[2 * x + 1] - b;
        if (n > SETUP_LONG) continue;
        uint16_t c[SETUP_LONG / 32];
        int rk[SETUP_LONG / 32];
#pragma unroll
        for (int i = 0; i < SETUP_LONG / 32; ++i) {
            c[i] = lane + 32 * i < n ? m.u.cval[b + lane + 32 * i] : 0;
            rk[i] = 0;
        }
        for (int y = 0; y < n; ++y) {
            const uint16_t o = m.u.cval[b + y];
#pragma unroll
            for (int i = 0; i < SETUP_LONG / 32; ++i) rk[i] += o < c[i];
        }
#pragma unroll
        for (int i = 0; i < SETUP_LONG / 32; ++i)
            if (lane + 32 * i < n) a.v2[b + rk[i]] = c[i];
    }
    for (int x = 0; x < nl; ++x) {
        const int b = m.pos[2 * x], n = m.pos[2 * x + 1] - b;
        if (n <= SETUP_LONG) continue;
        constexpr int W = 4 * SETUP_CTA_K / 32;
        if (tid < W) m.bits[tid] = 0u;
        __syncthreads();
        for (int y = tid; y < n; y += SETUP_CTA_THREADS) {
            const unsigned c = m.u.cval[b + y];
            atomicOr(&m.bits[c >> 5], 1u << (c & 31));
        }
        __syncthreads();
        unsigned word = tid < W ? m.bits[tid] : 0u, all;
        unsigned o = (unsigned)b + setup_cta_scan<false>((unsigned)__popc(word), m.ws, flip, all);
        while (word) {
            a.v2[o++] = 32 * tid + __ffs(word) - 1;
            word &= word - 1u;
        }
    }
}

// the rows of an indexed setup: gathered in the zones' order, and the
// groups' inverse blocks (float64, from the rows as assembled)
__device__ __forceinline__ void setup_rows(const SetupArgs &a, int k) {
    // a warp's share: consecutive warps of work on different CTAs (float64 is
    // slow on one SM)
    const int nw = gridDim.x * (blockDim.x >> 5), wi = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    for (int t = 32 * wi + (threadIdx.x & 31); t < k; t += 32 * nw) {
        const int src = a.zsrc[t];
        a.ids[t] = a.ids_raw[src];
        a.n64[t] = a.n64_raw[src];
        a.n32[t] = a.n32_raw[src];
        a.b[t] = a.b_raw[src];
    }
    group_inverses<PlainLd>(0, wi, nw, *a.d_ng, a.gst, a.ids_raw, a.n64_raw, a.nA,
                            a.wA, a.wB, a.pinv, a.zsrc);
}

constexpr int SETUP_ROWS_THREADS = 64;

__global__ void __launch_bounds__(SETUP_ROWS_THREADS) k_setup_rows(SetupArgs a) {
    HFCR_PDL_WAIT();
    setup_rows(a, max(0, min(*a.d_k, a.cap)));
}

union SetupSmem {
    SortSmem sort;
    int par[SETUP_SMALL_K];
};

__global__ void __launch_bounds__(TPB) k_setup(SetupArgs a) {
    HFCR_PDL_WAIT();
    const int k = max(0, min(*a.d_k, a.cap));
    if (a.indexed && k <= SETUP_CTA_K) {
        setup_rows(a, k);
        return;
    }
    // CTAs taking part: every CTA on large inputs, one per 1,024 entries on
    // small ones (the others leave at once; every CTA reads the same count)
    unsigned parts = gridDim.x;
    if (k <= SETUP_SMALL_K) {
        const unsigned want = (unsigned)max(1, (4 * k + SETUP_ENTRIES_PER_CTA - 1) / SETUP_ENTRIES_PER_CTA);
        if (want < parts) parts = want;
    }
    if (blockIdx.x >= parts) {
        if (k > 0) setup_helper(a, (int)parts);
        return;
    }
    __shared__ SetupSmem sh;
    SetupSync g{a.bar, 0u, a.status, parts};
    setup_phases(g, a, k, sh.sort, sh.par);
}

}  // namespace

void assemble(const MeshPair &mp, const hfcr_stencil *st, const int *d_k, int cap, double d,
              SolveBuffers &sb, uint32_t *d_status, cudaStream_t s) {
    if (cap <= 0) return;
    // dwork[8] / dwork[9]: the largest |b| and |dx| of the call, as the
    // bits of non-negative doubles
    { launch_pdl(k_assemble, (cap + 255) / 256, 256, 0, s, mp.A, mp.B, st, d_k, cap, d, sb.ids_raw,
                 sb.n64_raw, sb.n32_raw, sb.b_raw, (unsigned long long *)(sb.dwork + 8),
                 d_status); note_launch(); }
}

// dynamic shared memory granted to the zone CG kernels (0: the global-memory
// path runs); set once per process, outside any stream capture
static int g_fast_smem = -1, g_zone_pair_smem = 0, g_warp_zone_smem = 0;
static int g_rescue_smem = 0;  // of k_cg_zone64<true> (0: every zone on global memory)
static bool g_setup_cta = false;  // k_setup_cta has its shared memory
static bool g_cluster_ok = false;  // k_cg_zone_cl can be launched on this device

void solver_init() {
    if (g_fast_smem >= 0) return;
    g_fast_smem = cudaFuncSetAttribute(k_cg_zone<BIG_ZONE_THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       FAST_SMEM) == cudaSuccess ? FAST_SMEM : 0;
    if (!g_fast_smem) cudaGetLastError();
    g_zone_pair_smem = cudaFuncSetAttribute(k_cg_zone_pair, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            ZONE_PAIR_SMEM) == cudaSuccess ? ZONE_PAIR_SMEM : 0;
    if (!g_zone_pair_smem) cudaGetLastError();
    const int wz = WARP_ZONE_WARPS * WARP_ZONE_SMEM;
    g_warp_zone_smem = cudaFuncSetAttribute(k_cg_zone_warp, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            wz) == cudaSuccess ? wz : 0;
    if (!g_warp_zone_smem) cudaGetLastError();
    g_rescue_smem = cudaFuncSetAttribute(k_cg_zone64<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         RESCUE_SMEM) == cudaSuccess ? RESCUE_SMEM : 0;
    if (!g_rescue_smem) cudaGetLastError();
    g_setup_cta = cudaFuncSetAttribute(k_setup_cta, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       sizeof(SetupCtaSmem)) == cudaSuccess;
    if (!g_setup_cta) cudaGetLastError();
    // the cluster solver of large zones: its shared memory, and whether a
    // cluster of CL such CTAs fits on this device at all
    g_cluster_ok = false;
    if (cudaFuncSetAttribute(k_cg_zone_cl, cudaFuncAttributeMaxDynamicSharedMemorySize, CL_SMEM) ==
        cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(CL);
        cfg.blockDim = dim3(CL_THREADS);
        cfg.dynamicSmemBytes = CL_SMEM;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = CL;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int ncl = 0;
        g_cluster_ok = cudaOccupancyMaxActiveClusters(&ncl, (const void *)k_cg_zone_cl, &cfg) ==
                           cudaSuccess && ncl > 0;
    }
    cudaGetLastError();
}

// co-resident CTAs of k_setup on this device (0: cooperative launch unavailable)
static int setup_grid_max() {
    static int g[64] = {0};
    static bool done[64] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (!done[dev]) {
        int per_sm = 0, sms = 0, coop = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_setup, TPB, 0) == cudaSuccess &&
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop)
            // two CTAs per SM at most: the grid-wide phases are short and
            // every barrier costs one arrival per CTA
            g[dev] = (per_sm < 2 ? per_sm : 2) * sms;
        else
            cudaGetLastError();
        done[dev] = true;
    }
    return g[dev];
}

// the whole setup: up to SETUP_CTA_K stencils by k_setup_cta and a grid over
// the rows, above in one cooperative launch (which is then also the rows'
// grid, when the count turns out small); false when it cannot be launched
static bool build_setup_fused(const MeshPair &mp, const int *d_k, int cap, SolveBuffers &sb,
                              SortTemp &t, int *d_n4, uint32_t *d_status, cudaStream_t s) {
    if (!d_status || t.max_blocks < 3) return false;
    const bool small = g_setup_cta && cap <= SETUP_CTA_K;
    int grid = small ? 1 : setup_grid_max();
    if (grid <= 0) return false;
    const int tiles = (4 * cap + TILE - 1) / TILE;
    if (grid > tiles) grid = tiles > 0 ? tiles : 1;
    SetupArgs a;
    const int vb = bits_for((long long)mp.A.n_verts + mp.B.n_verts);
    a.d_k = d_k;
    a.cap = cap;
    a.vbits = 8 * ((vb + 7) / 8);
    a.nA = mp.A.n_verts;
    a.wA = mp.A.inv_mass;
    a.wB = mp.B.inv_mass;
    a.ids_raw = sb.ids_raw;
    a.n64_raw = sb.n64_raw;
    a.n32_raw = sb.n32_raw;
    a.b_raw = sb.b_raw;
    a.ckey = sb.ckey;
    a.ckey_alt = sb.ckey_alt;
    a.cflag = sb.cflag;
    a.cval = sb.cval;
    a.cval_alt = sb.cval_alt;
    a.zlab = (unsigned *)sb.zkey;
    a.zlab_alt = (unsigned *)sb.zkey_alt;
    a.zsrc = (int *)sb.zkey + cap;
    a.zsrc_alt = (int *)sb.zkey_alt + cap;
    a.k2 = (unsigned *)sb.ck64;
    a.k2_alt = (unsigned *)sb.ck64_alt;
    a.v2 = (int *)sb.ck64 + 4 * (size_t)cap;
    a.v2_alt = (int *)sb.ck64_alt + 4 * (size_t)cap;
    a.parent = sb.parent;
    a.ids = sb.ids;
    a.n64 = sb.n64;
    a.n32 = sb.n32;
    a.b = sb.b;
    a.szone = sb.szone;
    a.zs = sb.zs;
    a.zv = sb.zv;
    a.gst = sb.gst;
    a.zg = sb.zg;
    a.seg = sb.seg;
    a.gvert = sb.gvert;
    a.vidx = sb.vidx;
    a.winv = sb.winv;
    a.pinv = sb.pinv;
    a.d_n4 = d_n4;
    a.d_U = sb.d_U;
    a.d_nz = sb.d_nz;
    a.d_ng = sb.d_ng;
    a.hist = t.hist;
    a.tot = t.hist + 256 * (size_t)(t.max_blocks - 1);
    a.bar = t.hist + 256 * (size_t)(t.max_blocks - 2);
    a.status = d_status;
    a.indexed = g_setup_cta ? 1 : 0;
    if (g_setup_cta) {
        { launch_pdl(k_setup_cta, 1, SETUP_CTA_THREADS, sizeof(SetupCtaSmem), s, a); note_launch(); }
    } else {
        cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned), s);  // barrier counter, ready flag
    }
    sb.cval_s = a.v2;
    if (small) {
        { launch_pdl(k_setup_rows, (4 * cap + SETUP_ROWS_THREADS - 1) / SETUP_ROWS_THREADS, SETUP_ROWS_THREADS,
                     0, s, a); note_launch(); }
        return true;
    }
    void *args[] = {&a};
    if (cudaLaunchCooperativeKernel((const void *)k_setup, grid, TPB, args, 0, s) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    note_launch();
    return true;
}

void build_vertex_csr(const MeshPair &mp, const int *d_k, int cap, SolveBuffers &sb, SortTemp &t,
                      int *d_n4, uint32_t *d_status, int path, cudaStream_t s) {
    if (cap <= 0) return;
    if (path == 0 && build_setup_fused(mp, d_k, cap, sb, t, d_n4, d_status, s)) return;
    // the same setup as a sequence of kernels
    int n4 = 4 * cap;
    int nb = (n4 + 255) / 256;
    int gb = (cap + 255) / 256;
    if (gb > 1024) gb = 1024;
    // vertex -> stencils of the rows as assembled (for the impact zones)
    { launch_pdl(k_csr_entries, nb, 256, 0, s, sb.ids_raw, d_k, cap, sb.ckey,
                 sb.cval); note_launch(); }
    { launch_pdl(k_csr_flags, 1, 1, 0, s, sb.ckey, d_k, cap, sb.cflag,
                 d_n4); note_launch(); }  // count only
    int vb = bits_for((long long)mp.A.n_verts + mp.B.n_verts);
    bool flip = radix_sort_u32_dev(sb.ckey, sb.cval, sb.ckey_alt, sb.cval_alt, d_n4, n4, vb, t, s);
    unsigned *ck1 = flip ? sb.ckey_alt : sb.ckey;
    int *cv1 = flip ? sb.cval_alt : sb.cval;
    { launch_pdl(k_csr_flags, nb, 256, 0, s, ck1, d_k, cap, sb.cflag, d_n4); note_launch(); }
    scan_flags_dev(sb.cflag, d_n4, n4, sb.d_U, t, s);
    { launch_pdl(k_csr_build, nb, 256, 0, s, ck1, cv1, sb.cflag, d_k, cap, mp.A.n_verts,
                 mp.A.inv_mass,
                                   mp.B.inv_mass, sb.vidx, sb.seg, sb.gvert, sb.winv); note_launch(); }
    // impact zones and the zone-ordered rows.  The 64-bit scratch arrays
    // are used as pairs of 32-bit arrays: (label, stencil) for the zone sort,
    // (zone, entry) for the zone-ordered CSR.
    int kb = bits_for((long long)cap + 1);
    unsigned *zlab = (unsigned *)sb.zkey, *zlab_alt = (unsigned *)sb.zkey_alt;
    int *zsrc = (int *)sb.zkey + cap, *zsrc_alt = (int *)sb.zkey_alt + cap;
    { launch_pdl(k_uf_small, 1, 1024, 0, s, d_k, sb.d_U, sb.seg, cv1, zlab, zsrc,
                 d_status); note_launch(); }
    if (cap > UF_SMALL) {
        { launch_pdl(k_uf_init, gb, 256, 0, s, d_k, sb.parent); note_launch(); }
        { launch_pdl(k_uf_union, nb < 1024 ? nb : 1024, 256, 0, s, d_k, sb.d_U, sb.seg, cv1,
                     sb.parent, d_status); note_launch(); }
        { launch_pdl(k_zone_keys, gb, 256, 0, s, d_k, sb.parent, zlab, zsrc); note_launch(); }
    }
    bool zflip = radix_sort_u32_dev(zlab, zsrc, zlab_alt, zsrc_alt, d_k, cap, kb, t, s);
    unsigned *zl = zflip ? zlab_alt : zlab;
    int *zr = zflip ? zsrc_alt : zsrc;
    { launch_pdl(k_zone_flags, gb, 256, 0, s, d_k, zl, sb.cflag); note_launch(); }
    scan_flags_dev(sb.cflag, d_k, cap, sb.d_nz, t, s);
    int *pos_of = sb.parent;  // the forest is no longer needed
    { launch_pdl(k_zone_gather, gb, 256, 0, s, d_k, zl, zr, sb.cflag, sb.ids_raw, sb.n64_raw,
                 sb.n32_raw,
                                     sb.b_raw, sb.ids, sb.n64, sb.n32, sb.b, sb.szone, sb.zs,
                                     pos_of); note_launch(); }
    // vertex-ordered entries re-sorted stably by zone: zone-contiguous numbering
    unsigned *k2 = (unsigned *)sb.ck64, *k2_alt = (unsigned *)sb.ck64_alt;
    int *v2 = (int *)sb.ck64 + n4, *v2_alt = (int *)sb.ck64_alt + n4;
    { launch_pdl(k_csr2_entries, nb, 256, 0, s, cv1, pos_of, sb.szone, d_k, cap, k2,
                 v2); note_launch(); }
    bool flip2 = radix_sort_u32_dev(k2, v2, k2_alt, v2_alt, d_n4, n4, kb, t, s);
    unsigned *zk2 = flip2 ? k2_alt : k2;
    sb.cval_s = flip2 ? v2_alt : v2;
    { launch_pdl(k_csr2_flags, nb, 256, 0, s, sb.cval_s, sb.ids, d_k, cap,
                 sb.cflag); note_launch(); }
    scan_flags_dev(sb.cflag, d_n4, n4, sb.d_U, t, s);
    { launch_pdl(k_csr2_build, nb, 256, 0, s, zk2, sb.cval_s, sb.cflag, sb.ids, d_k, cap,
                 mp.A.n_verts,
                                    mp.A.inv_mass, mp.B.inv_mass, sb.vidx, sb.seg, sb.gvert, sb.winv,
                                    sb.zv, sb.d_nz); note_launch(); }
    // groups of rows sharing x0 and the inverses of their blocks
    { launch_pdl(k_group_flags, gb, 256, 0, s, d_k, sb.ids, sb.szone, sb.zs,
                 sb.cflag); note_launch(); }
    scan_flags_dev(sb.cflag, d_k, cap, sb.d_ng, t, s);
    { launch_pdl(k_group_build, gb, 256, 0, s, d_k, sb.ids, sb.szone, sb.zs, sb.cflag, sb.d_nz,
                 sb.gst,
                                     sb.zg); note_launch(); }
    { launch_pdl(k_group_inverse, gb, 128, 0, s, sb.d_ng, sb.gst, sb.ids, sb.n64, mp.A.n_verts,
                 mp.A.inv_mass, mp.B.inv_mass, sb.pinv); note_launch(); }
}

void solve(const SolveParams &p, const MeshPair &mp, const int *d_k, int cap, SolveBuffers &sb,
           uint32_t *d_status, cudaStream_t s) {
    (void)d_status;
    if (cap <= 0) return;
    solver_init();
    const int fast_smem = g_fast_smem;
    int rb = (cap + 255) / 256;
    if (rb > RES_BLOCKS) rb = RES_BLOCKS;
    // sb.iwork and sb.dwork were zeroed with the call's other device words
    if (p.solver == HFCR_SOLVER_FP64) {
        // the plain float64 form: every impact zone by its own CTA, float64
        // CG with the whole iteration budget of the mixed solver
        ZoneArgs za;
        za.zs = sb.zs; za.zv = sb.zv; za.zg = sb.zg;
        za.seg = sb.seg; za.cval = sb.cval_s; za.winv = sb.winv;
        za.n32 = sb.n32; za.pinv = sb.pinv; za.n64 = sb.n64; za.vidx = sb.vidx; za.gst = sb.gst;
        za.b64 = sb.b; za.lam = sb.lam; za.u64 = sb.u64; za.zres = sb.r64; za.zbb = sb.q64;
        za.maxit = p.max_cg_iters; za.max_refine = p.max_refine;
        za.tol = p.inner_tol; za.rel_tol = p.rel_tol; za.ctl = sb.iwork;
        za.ticket = (unsigned *)(sb.iwork + 13);
        za.ids = sb.ids;
        za.nA = mp.A.n_verts;
        za.wA = mp.A.inv_mass;
        za.wB = mp.B.inv_mass;
        za.pinv64 = sb.pinv64;
        Zone64Scratch g64;
        g64.r = sb.cg64; g64.p = sb.cg64 + cap; g64.s = sb.cg64 + 2 * (size_t)cap;
        g64.w = sb.cg64 + 3 * (size_t)cap; g64.z = sb.cg64 + 4 * (size_t)cap;
        int zg = cap < 4 * 152 ? cap : 4 * 152;
        { launch_pdl(k_cg_zone64<false>, zg, ZONE64_THREADS, 0, s, sb.d_nz, za, g64,
                     p.max_cg_iters * p.max_refine, 0); note_launch(); }
        { launch_pdl(k_zone_final, 1, 256, 0, s, sb.d_nz, sb.r64, sb.q64, p.rel_tol, sb.dwork,
                     sb.iwork); note_launch(); }
        return;
    }
    if (p.solver == HFCR_SOLVER_FP64_GLOBAL) {
        // one float64 run with the whole iteration budget of the mixed solver
        { launch_pdl(k_init_lam, rb, 256, 0, s, d_k, sb.b, sb.lam, sb.r64); note_launch(); }
        { launch_pdl(k_cg<double>, 1, CG_THREADS, 0, s, 1, d_k, sb.d_U, sb.seg, sb.cval_s,
                     sb.winv, sb.n64,
                                              sb.vidx, sb.b, sb.lam, sb.p64 + 0, sb.r64, sb.p64 + cap,
                                              sb.q64, sb.u64, p.max_cg_iters * p.max_refine,
                                              p.rel_tol, sb.iwork); note_launch(); }
        { launch_pdl(k_res_vertex, rb, 256, 0, s, sb.d_U, sb.seg, sb.cval_s, sb.winv, sb.n64,
                     sb.lam, sb.u64,
                                         sb.iwork); note_launch(); }
        { launch_pdl(k_res_stencil, rb, 256, 0, s, d_k, sb.vidx, sb.n64, sb.b, sb.u64, sb.r64,
                     sb.red,
                                          sb.iwork, (unsigned *)(sb.iwork + 12), p.rel_tol,
                                          sb.dwork, 0); note_launch(); }
        return;
    }
    // MIXED: float32 PCG with float64 refinement, each zone to convergence
    // in its own CTA.  r64 and q64 (float64 scratch of the FP64 solver) hold
    // the zones' final |r|^2 and |b|^2.
    ZoneArgs za;
    za.zs = sb.zs; za.zv = sb.zv; za.zg = sb.zg;
    za.seg = sb.seg; za.cval = sb.cval_s; za.winv = sb.winv;
    za.n32 = sb.n32; za.pinv = sb.pinv; za.n64 = sb.n64; za.vidx = sb.vidx; za.gst = sb.gst;
    za.b64 = sb.b; za.lam = sb.lam; za.u64 = sb.u64; za.zres = sb.r64; za.zbb = sb.q64;
    za.maxit = p.max_cg_iters; za.max_refine = p.max_refine;
    za.tol = p.inner_tol; za.rel_tol = p.rel_tol; za.ctl = sb.iwork;
    za.ticket = (unsigned *)(sb.iwork + 13);  // iwork is zeroed before every solve
    za.binv = sb.binv;
    za.block_switch = p.block_switch;
    const int warp_max = g_warp_zone_smem ? WARP_ZONE : 0;
    if (warp_max) {
        int zw = (cap + WARP_ZONE_WARPS - 1) / WARP_ZONE_WARPS;  // CTAs of the warp launch
        if (zw > 4 * 152) zw = 4 * 152;
        { launch_pdl(k_cg_zone_warp, zw, 32 * WARP_ZONE_WARPS, g_warp_zone_smem, s, sb.d_nz,
                     za); note_launch(); }
    }
    ZoneScratch gs;
    gs.x = sb.x32; gs.r = sb.r32; gs.p = sb.p32; gs.s = sb.q32; gs.w = sb.w32; gs.z = sb.z32;
    gs.u = sb.u32;
    // CTAs of the pair launch: two zones of more than warp_max stencils at
    // a time (at most 2 CTAs per SM); of the large-zone launch: one zone
    // of ZONE_BIG or more stencils each
    int zpair = (cap / (WARP_ZONE + 1) + 1) / 2 + 1;
    if (zpair > 2 * 152) zpair = 2 * 152;
    int zbig = (cap + ZONE_MID - 1) / ZONE_MID;
    if (zbig > 152) zbig = 152;
    { launch_pdl(k_cg_zone_pair, zpair, 512, g_zone_pair_smem, s, sb.d_nz, za, warp_max, gs,
                 g_zone_pair_smem, zbig); note_launch(); }
    // zones of ZONE_BIG rows or more: one CTA each when they fit its shared
    // memory; larger ones on a cluster of CL CTAs (or, without
    // clusters, on global memory)
    p.big_mark(1, s);
    { launch_pdl(k_cg_zone<BIG_ZONE_THREADS>, zbig, BIG_ZONE_THREADS, fast_smem, s, sb.d_nz, za, ZONE_BIG - 1,
                 ZONE_MID, gs, fast_smem, g_cluster_ok ? 1 : 0); note_launch(); }
    if (g_cluster_ok) {
        int ncl = (cap + ZONE_CL_MIN - 1) / ZONE_CL_MIN;
        if (ncl > 152 / CL) ncl = 152 / CL;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(ncl * CL);
        cfg.blockDim = dim3(CL_THREADS);
        cfg.dynamicSmemBytes = CL_SMEM;
        cfg.stream = s;
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = CL;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = 2;
        cudaLaunchKernelEx(&cfg, k_cg_zone_cl, (const int *)sb.d_nz, za, gs, fast_smem);
        note_launch();
    }
    p.big_mark(0, s);
    // a zone whose float32 runs stopped reducing its float64 residual before
    // the target (the residual guard) is solved again by the float64 per-zone
    // CG; every other zone is skipped at once
    za.ids = sb.ids;
    za.nA = mp.A.n_verts;
    za.wA = mp.A.inv_mass;
    za.wB = mp.B.inv_mass;
    za.pinv64 = sb.pinv64;
    {
        Zone64Scratch g64;
        g64.r = sb.cg64; g64.p = sb.cg64 + cap; g64.s = sb.cg64 + 2 * (size_t)cap;
        g64.w = sb.cg64 + 3 * (size_t)cap; g64.z = sb.cg64 + 4 * (size_t)cap;
        int zr = cap < 152 ? cap : 152;
        { launch_pdl(k_cg_zone64<true>, zr, RESCUE_THREADS, g_rescue_smem, s, sb.d_nz, za, g64,
                     p.max_cg_iters * p.max_refine, g_rescue_smem); note_launch(); }
    }
    { launch_pdl(k_zone_final, 1, 256, 0, s, sb.d_nz, sb.r64, sb.q64, p.rel_tol, sb.dwork,
                 sb.iwork); note_launch(); }
}

void displacement(const MeshPair &mp, int cap, SolveBuffers &sb, int apply, void *const *dxA,
                  void *const *dxB, cudaStream_t s) {
    if (cap <= 0) return;
    int nb = (4 * cap + 255) / 256;
    if (nb > 1024) nb = 1024;
    void *a0 = dxA ? dxA[0] : nullptr, *a1 = dxA ? dxA[1] : nullptr, *a2 = dxA ? dxA[2] : nullptr;
    void *b0 = dxB ? dxB[0] : nullptr, *b1 = dxB ? dxB[1] : nullptr, *b2 = dxB ? dxB[2] : nullptr;
    { launch_pdl(k_displace, nb, 256, 0, s, sb.d_U, sb.seg, sb.cval_s, sb.winv, sb.n64, sb.lam,
                 sb.gvert, mp.A, mp.B, apply, a0, a1, a2, b0, b1, b2,
                 (unsigned long long *)(sb.dwork + 9)); note_launch(); }
}

}  // namespace hfcr
