// Element Jacobians k_e = d r_e / d u_e (the 32 x 32 element matrix of Algorithm 4, before the
// hanging correction M_e^T k_e M_e of Algorithm 2) and the nodal block-Jacobi diagonal.
//
// Every column of k_e is the derivative of the element residual in the direction of one local
// degree of freedom (corner b, component k).  The fields of the point are interpolated once
// (values); the seed's tangent fields are read off the basis of corner b at the point, then the
// pointwise VMS coefficients are differentiated exactly (dual numbers), weighted and contracted
// with the test functions.  No global matrix is ever formed.
//
//   float64: jac_out64, jac_cut64, jac_surf64 (lane = column of k_e); float32 element arithmetic:
//   jac_out     8 threads per Out element (thread c: Gauss point c, then node c's 4 rows)
//   jac_cut     four warps per Intercepted element, 32 sub-cell points per step, lane = point, then row
//   jac_nitsche one thread per surface point (a warp per block: there are few points, and each is long)
// Mode FULL writes k_e for requested elements (slot map); mode DIAG adds the 4x4 diagonal blocks
// of sum_e M_e^T k_e M_e (each corner's own block times the squared hanging weights; the
// couplings of two different corners of one element that share a parent are left out) to a
// float64 [n_nodes][4][4] array.

#include <cuda_runtime.h>

#include "imga_internal.h"
#include "vms_device.cuh"

namespace imga {

namespace {

enum { FULL = 0, DIAG = 1, BSR = 2 };

// Position of block (row, col) in the block pattern (columns increasing within a row), or -1.
__device__ __forceinline__ int64_t bsr_find(const int64_t* __restrict__ ptr, const int32_t* __restrict__ idx,
                                            int32_t row, int32_t col) {
    int64_t lo = ptr[row], hi = ptr[row + 1] - 1;
    while (lo <= hi) {
        const int64_t mid = (lo + hi) >> 1;
        const int32_t c = idx[mid];
        if (c == col) return mid;
        if (c < col) lo = mid + 1;
        else hi = mid - 1;
    }
    return -1;
}

// node ids and weights a corner enters through M_e: itself, or the 2 / 4 parents of a hanging node
__device__ __forceinline__ int corner_nodes(const Args& A, int32_t id, int32_t nd[4], double& w) {
    if (id < A.n_nodes) { nd[0] = id; w = 1.0; return 1; }
    const int32_t* hp = A.hpar + 4 * (int64_t)(id - A.n_nodes);
    const int np = hp[2] >= 0 ? 4 : 2;
    for (int p = 0; p < np; ++p) nd[p] = hp[p];
    w = np == 4 ? 0.25 : 0.5;
    return np;
}

// N entries of row or block (corner ida, corner idb) of k_e added to the assembled matrix through
// M_e^T k_e M_e (Algorithm 2): every parent pair (p, q) receives w_p w_q v in block (p, q), entry at[j]
// (4 x row component + column component).  The row is searched once per corner pair: entry by entry the
// searches were most of the assembly (43.6 k elements,
// mixed: 5.37 -> 1.45 ms with the basis tables, the shared test functions, the adds below and selected seeds).
// A warp adds whole blocks from shared memory where it can (bsr_add_blocks): 16 lanes on the 128 bytes of a
// block make 4 L2 transactions of what lane-by-lane adds make 16 of.
// Float entries are weighted (powers of two: exact) and tested in float32 and widened on the integer pipe:
// the FP64 pipe was 58 % busy with that alone.
__device__ __forceinline__ double wide(float x) { return f2d(x); }
__device__ __forceinline__ double wide(double x) { return x; }
template <int N, class T, class At>
__device__ __forceinline__ void bsr_add(const Args& A, int32_t ida, int32_t idb, const T* v, At at, double* __restrict__ val) {
    int32_t na[4], nb[4];
    double wa, wb;
    const int ca = corner_nodes(A, ida, na, wa), cb = corner_nodes(A, idb, nb, wb);
    const T w = (ca == 1 ? T(1) : ca == 2 ? T(0.5) : T(0.25)) * (cb == 1 ? T(1) : cb == 2 ? T(0.5) : T(0.25));
    for (int p = 0; p < ca; ++p)
        for (int q = 0; q < cb; ++q) {
            const int64_t pos = bsr_find(A.bptr, A.bidx, na[p], nb[q]);
            if (pos < 0) continue;
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (v[j] != T(0)) atomicAdd(val + 16 * pos + at(j), wide(w * v[j]));
        }
}

// N blocks by a warp, entry (block m, j) given by v(m, j), to positions s_pos[m] (-1: none)
template <int N, class V>
__device__ __forceinline__ void bsr_add_blocks(const int64_t* s_pos, V v, int lane, double* __restrict__ val) {
#pragma unroll 4
    for (int m = lane >> 4; m < N; m += 2) {
        const int64_t pos = s_pos[m];
        const auto x = v(m, lane & 15);
        if (pos >= 0 && x != 0) atomicAdd(val + 16 * pos + (lane & 15), wide(x));
    }
}
__device__ __forceinline__ bool plain_corner(const Args& A, int32_t id) { return id < A.n_nodes; }

// The block (corner ida, corner idb) of a warp's element, at least one of them hanging, through M_e: lane 4 p + q
// searches the block of parent pair (p, q), then 16 lanes add each pair's 16 entries v(j).  Uniform call.
template <class V>
__device__ __forceinline__ void bsr_add_hanging(const Args& A, int32_t ida, int32_t idb, V v, int lane, double* __restrict__ val) {
    const int p = (lane >> 2) & 3, q = lane & 3;
    auto node = [&](int32_t id, int k, int& n) -> int32_t {   // k-th node of a corner and how many there are
        if (id < A.n_nodes) { n = 1; return id; }
        const int32_t* hp = A.hpar + 4 * (int64_t)(id - A.n_nodes);
        n = hp[2] >= 0 ? 4 : 2;
        return k < n ? hp[k] : -1;
    };
    int ca, cb;
    const int32_t row = node(ida, p, ca), col = node(idb, q, cb);
    const int64_t pos = lane < 16 && p < ca && q < cb ? bsr_find(A.bptr, A.bidx, row, col) : -1;
    const auto x = v(lane & 15);
    const auto w = x * (ca == 1 ? 1.f : ca == 2 ? 0.5f : 0.25f) * (cb == 1 ? 1.f : cb == 2 ? 0.5f : 0.25f);
    const double d = wide(w);
#pragma unroll 1
    for (int m = 0; m < 16; m += 2) {
        if (((m >> 2) >= ca) || (m & 3) >= cb) continue;   // uniform (pairs m, m + 1: q even and odd)
        const int64_t o = __shfl_sync(0xffffffffu, pos, m + (lane >> 4));
        if (o >= 0 && x != 0) atomicAdd(val + 16 * o + (lane & 15), d);
    }
}

// tangent fields of the seed (corner b, component k) at a point whose corner-b basis values are
// phb, reference gradient dphb and reference mixed second derivatives d2b (01, 02, 12)
template <class T>
__device__ __forceinline__ void seed_fields(const Args& A, const Fields<T, T>& V, T g, T phb, const T dphb[3],
                                            const T d2b[3], int k, Fields<Dual<T>, T>& F) {
    // (k is known only at run time, so tangents are selected: an indexed store would put F in local memory)
    const T th = (T)A.theta, c0 = (T)A.c0, g2 = g * g;
    const T tu = th * phb, ta = c0 * phb;
    T tg[3], tp[3], th2[3];
    for (int j = 0; j < 3; ++j) { tg[j] = th * g * dphb[j]; tp[j] = g * dphb[j]; th2[j] = th * g2 * d2b[j]; }
    const bool vel = k < 3;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const bool own = i == k;
        F.us[i] = {V.us[i], own ? tu : T(0)};
        F.at[i] = {V.at[i], own ? ta : T(0)};
        F.gp[i] = {V.gp[i], vel ? T(0) : tp[i]};
        // (grad div u)_i = sum_{j != i} d_i d_j u_j: a unit u_k at corner b feeds every i != k, by pair (i, k)
        // (xy, xz, yz: 0, 1, 2)
        const T h = i == 0 ? (k == 1 ? th2[0] : th2[1]) : i == 1 ? (k == 0 ? th2[0] : th2[2]) : (k == 0 ? th2[1] : th2[2]);
        F.H2[i] = {V.H2[i], vel && !own ? h : T(0)};
        F.f[i] = V.f[i];
#pragma unroll
        for (int j = 0; j < 3; ++j) F.Gu[i][j] = {V.Gu[i][j], own ? tg[j] : T(0)};
    }
    F.p = {V.p, vel ? T(0) : phb};
}

template <class T>
__device__ __forceinline__ void corner_basis(const T fm[3], const T fp[3], int b, T& ph, T dph[3], T d2[3]) {
    const T f0 = (b & 1) ? fp[0] : fm[0], f1 = (b & 2) ? fp[1] : fm[1], f2 = (b & 4) ? fp[2] : fm[2];
    const T h0 = (b & 1) ? T(0.5) : T(-0.5), h1 = (b & 2) ? T(0.5) : T(-0.5), h2 = (b & 4) ? T(0.5) : T(-0.5);
    ph = f0 * f1 * f2;
    dph[0] = h0 * (f1 * f2);
    dph[1] = h1 * (f0 * f2);
    dph[2] = h2 * (f0 * f1);
    d2[0] = (h0 * h1) * f2;
    d2[1] = (h0 * h2) * f1;
    d2[2] = (h1 * h2) * f0;
}

// add a corner's 4x4 block to the diagonal of its node(s) through the hanging weights
__device__ __forceinline__ void add_diag(const Args& A, int32_t id, const double blk[16], double* D) {
    if (id < A.n_nodes) {
        for (int q = 0; q < 16; ++q) atomicAdd(D + 16 * (int64_t)id + q, blk[q]);
        return;
    }
    const int32_t* hp = A.hpar + 4 * (int64_t)(id - A.n_nodes);
    const int np = hp[2] >= 0 ? 4 : 2;
    const double w2 = np == 4 ? 0.0625 : 0.25;
    for (int p = 0; p < np; ++p)
        for (int q = 0; q < 16; ++q) atomicAdd(D + 16 * (int64_t)hp[p] + q, w2 * blk[q]);
}

constexpr int kOutEpb = 16;   // Out elements per block

// Bound by issue and dependent chains.  The seeds are selected (see seed_fields), as an indexed store would put 240
// bytes per thread in local memory; only the diagonal form keeps an array there (144 bytes of stack).  Registers for
// five blocks per SM (8 to 40 bytes of spills): 2.8 waves instead of 3.5 on 33.7 k Out elements.  An assembly of 43.6 k
// elements 1,858 -> 1,505 us with the selected seeds here and in jac_cut, 1,450 with the fifth block and the
// 16-byte accesses below.
template <int MODE>
__global__ void __launch_bounds__(8 * kOutEpb, 5) jac_out(Args A, const int32_t* __restrict__ list, int64_t n,
                                                          const int32_t* __restrict__ slot, double* __restrict__ K,
                                                          double* __restrict__ D) {
    typedef float T;
    constexpr int EPB = kOutEpb;
    __shared__ __align__(16) T s_nd[EPB][8][CS];
    // a Gauss point's coefficients, in fours (component i: phi and gradient coefficients), for 16-byte accesses;
    // the strides keep the four elements of a warp, and its points, on different banks
    __shared__ __align__(16) T s_cf[EPB][8 * 20 + 4];
    __shared__ __align__(16) T s_bas[8][8][4];   // [Gauss point q][corner c]: phi, reference gradient
    __shared__ T s_blk[MODE == BSR ? EPB / 4 : 1][32][17];      // BSR: block (corner c, corner b) of every lane
    __shared__ int64_t s_pos[MODE == BSR ? EPB / 4 : 1][32];
    const int c = threadIdx.x & 7, le = threadIdx.x >> 3;
    for (int t = threadIdx.x; t < 64; t += blockDim.x) {   // the same for every element and seed
        const T gs = (T)0.57735026918962576451;
        const T wp = T(0.5) * (T(1) + gs), wm = T(0.5) * (T(1) - gs);
        const int q = t >> 3, cc = t & 7;
        T f[3], d[3];
        for (int kk = 0; kk < 3; ++kk) {
            const bool same = (((cc >> kk) & 1) == ((q >> kk) & 1));
            f[kk] = same ? wp : wm;
            d[kk] = ((cc >> kk) & 1) ? T(0.5) : T(-0.5);
        }
        s_bas[q][cc][0] = f[0] * f[1] * f[2];
        s_bas[q][cc][1] = d[0] * f[1] * f[2];
        s_bas[q][cc][2] = d[1] * f[0] * f[2];
        s_bas[q][cc][3] = d[2] * f[0] * f[1];
    }
    __syncthreads();
    const int64_t idx = (int64_t)blockIdx.x * EPB + le;
    const bool valid = idx < n;
    const int32_t e = list[valid ? idx : n - 1];
    const int32_t sl = MODE == FULL ? slot[e] : 0;
    const bool work = valid && sl >= 0;
    const int32_t id = A.conn[8 * (int64_t)e + c];
    corner_data<T, false>(A, id, &s_nd[le][c][0]);
    __syncwarp();
    const int lv = A.lev[e];
    const T g = lvl_g<T>(A, lv);
    const T gauss = (T)0.57735026918962576451;
    const T wp = T(0.5) * (T(1) + gauss), wm = T(0.5) * (T(1) - gauss);
    T fm[3], fp[3];
    for (int k = 0; k < 3; ++k) {
        const bool plus = (c >> k) & 1;
        fm[k] = plus ? wm : wp;
        fp[k] = plus ? wp : wm;
    }
    Fields<T, T> V;
    interp<T, T>(A, fm, fp, &s_nd[le][0][0], CS, g, V);
    const T wq = lvl_w<T>(A, lv), wqg = wq * g;
    double diag[16];
    for (int q = 0; q < 16; ++q) diag[q] = 0.0;
    for (int b = 0; b < 8; ++b) {
        T phb, dphb[3], d2b[3];
        corner_basis<T>(fm, fp, b, phb, dphb, d2b);
#pragma unroll 1   // (unrolled, the shared value part is contracted differently: other last bits)
        for (int k = 0; k < 4; ++k) {
            Fields<Dual<T>, T> F;
            seed_fields<T>(A, V, g, phb, dphb, d2b, k, F);
            Dual<T> cf[16];
            pointwise<Dual<T>, T>(A, Phys<T>(A, prob_of(A, e)), F, g, cf);
            T cw[16];
            for (int q = 0; q < 16; ++q) cw[q] = ((q < 3 || q == 12) ? wq : wqg) * cf[q].d;
            for (int i = 0; i < 3; ++i) st4s<T>(&s_cf[le][20 * c + 4 * i], cw[i], cw[3 + 3 * i], cw[4 + 3 * i], cw[5 + 3 * i]);
            st4s<T>(&s_cf[le][20 * c + 12], cw[12], cw[13], cw[14], cw[15]);
            __syncwarp();
            T r[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                T bs[4];
                ld4s<T>(&s_bas[q][c][0], bs);
                const T ph = bs[0];
                const T* dp = bs + 1;
                for (int i = 0; i < 4; ++i) {
                    T C[4];
                    ld4s<T>(&s_cf[le][20 * q + 4 * i], C);
                    r[i] += ph * C[0] + dp[0] * C[1] + dp[1] * C[2] + dp[2] * C[3];
                }
            }
            __syncwarp();
            if (MODE == FULL) {
                if (work)
                    for (int i = 0; i < 4; ++i) K[(int64_t)sl * 1024 + (c * 4 + i) * 32 + b * 4 + k] = (double)r[i];
            } else if (MODE == BSR) {
                for (int i = 0; i < 4; ++i) s_blk[threadIdx.x >> 5][threadIdx.x & 31][i * 4 + k] = r[i];
            } else if (b == c) {
                for (int i = 0; i < 4; ++i) diag[i * 4 + k] = (double)r[i];
            }
        }
        if (MODE == BSR) {
            const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
            const int32_t idb = __shfl_sync(0xffffffffu, id, (lane & ~7) | b);
            const bool plain = plain_corner(A, id) && plain_corner(A, idb);
            s_pos[w][lane] = work && plain ? bsr_find(A.bptr, A.bidx, id, idb) : -1;
            __syncwarp();
            bsr_add_blocks<32>(s_pos[w], [&](int m, int j) { return s_blk[w][m][j]; }, lane, K);
            for (unsigned need = __ballot_sync(0xffffffffu, work && !plain); need; need &= need - 1) {
                const int src = __ffs(need) - 1;
                const int32_t ha = __shfl_sync(0xffffffffu, id, src), hb = __shfl_sync(0xffffffffu, idb, src);
                bsr_add_hanging(A, ha, hb, [&](int j) { return s_blk[w][src][j]; }, lane, K);
            }
            __syncwarp();
        }
    }
    if (MODE == DIAG && work) add_diag(A, id, diag, D);
}

constexpr int JWPB = 4;   // warps per element of jac_cut

// An Intercepted element: a block of four warps, lane = sub-cell point (32 at a time), each warp the seeds
// of two corners.  A warp alone with an element ran its hundreds of points 32 seeds deep while most of the
// chip had nothing left (7.3 k element sphere, 776 elements: 660 -> 361 us an assembly).
template <int MODE>
__global__ void __launch_bounds__(32 * JWPB) jac_cut(Args A, const int32_t* __restrict__ list,
                                                     const int64_t* __restrict__ off, const void* __restrict__ pts,
                                                     const int32_t* __restrict__ order, const int32_t* __restrict__ slot,
                                                     double* __restrict__ K, double* __restrict__ D) {
    typedef float T;
    constexpr int NB = 8 / JWPB;                    // corners (of the seeds) per warp
    __shared__ __align__(16) T s_nd[8][CS];
    // a point's coefficients for the four seeds of a corner, in fours (component c: phi and gradient
    // coefficients) at place c ^ (point / 2 & 3): conflict-free 16-byte stores.  The contraction, bound by shared
    // memory, reads a point's test functions once for four sums.
    __shared__ __align__(16) T s_cf[JWPB][4][32][16];
    __shared__ __align__(16) T s_bas[32][8][4];     // a point's test functions (phi, reference gradient), once for all seeds
    __shared__ T s_acc[32][32];                     // the element's columns so far
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t idx = order[blockIdx.x];
    const int32_t e = list[idx];
    const int32_t sl = MODE == FULL ? slot[e] : 0;
    if (sl < 0) return;
    int32_t my_id = 0;
    if (lane < 8) {
        my_id = A.conn[8 * (int64_t)e + lane];
        if (w == 0) corner_data<T, false>(A, my_id, &s_nd[lane][0]);
    }
    __syncthreads();
    const T g = lvl_g<T>(A, A.lev[e]);
    const T det = lvl_w<T>(A, A.lev[e]);
    const int a = lane >> 2, comp = lane & 3;
    T* acc = &s_acc[0][lane];   // acc[32 s]: row `lane` of column s
    for (int s = 4 * NB * w; s < 4 * NB * (w + 1); ++s) acc[32 * s] = T(0);
    const int64_t q0 = off[idx], q1 = off[idx + 1];
    for (int64_t base = q0; base < q1; base += 32) {
        const int64_t q = base + lane;
        const bool have = q < q1;
        T pt[4] = {T(0), T(0), T(0), T(0)};
        if (have) load_pt<T>(pts, q, pt);
        T fm[3], fp[3];
        for (int k = 0; k < 3; ++k) { fm[k] = T(0.5) * (T(1) - pt[k]); fp[k] = T(0.5) * (T(1) + pt[k]); }
        Fields<T, T> V;
        interp<T, T>(A, fm, fp, &s_nd[0][0], CS, g, V);
        const T wq = have ? pt[3] * det : T(0), wqg = wq * g;
        const int m = (int)min((int64_t)32, q1 - base);
        for (int cc = NB * w; cc < NB * (w + 1); ++cc) {
            const T s0 = (cc & 1) ? T(1) : T(-1), s1 = (cc & 2) ? T(1) : T(-1), s2 = (cc & 4) ? T(1) : T(-1);
            const T f0 = T(0.5) * (T(1) + s0 * pt[0]), f1 = T(0.5) * (T(1) + s1 * pt[1]), f2 = T(0.5) * (T(1) + s2 * pt[2]);
            st4s<T>(&s_bas[lane][cc][0], f0 * f1 * f2, T(0.5) * s0 * f1 * f2, T(0.5) * s1 * f0 * f2, T(0.5) * s2 * f0 * f1);
        }
        __syncthreads();
        for (int b = NB * w; b < NB * (w + 1); ++b) {
            T phb, dphb[3], d2b[3];
            corner_basis<T>(fm, fp, b, phb, dphb, d2b);
#pragma unroll 1   // as in jac_out
            for (int k = 0; k < 4; ++k) {
                Fields<Dual<T>, T> F;
                seed_fields<T>(A, V, g, phb, dphb, d2b, k, F);
                Dual<T> cf[16];
                pointwise<Dual<T>, T>(A, Phys<T>(A, prob_of(A, e)), F, g, cf);
                T cw[16];
                for (int qq = 0; qq < 16; ++qq) cw[qq] = ((qq < 3 || qq == 12) ? wq : wqg) * cf[qq].d;
                T* dst = &s_cf[w][k][lane][0];
                const int x = (lane >> 1) & 3;
                for (int i = 0; i < 3; ++i) st4s<T>(dst + 4 * (i ^ x), cw[i], cw[3 + 3 * i], cw[4 + 3 * i], cw[5 + 3 * i]);
                st4s<T>(dst + 4 * (3 ^ x), cw[12], cw[13], cw[14], cw[15]);
            }
            __syncwarp();
            T sum[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll 2
            for (int j = 0; j < m; ++j) {
                T B[4];
                ld4s<T>(&s_bas[j][a][0], B);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    // (multiply-adds spelled out: contracted otherwise, the sum has other last bits)
                    T C[4];
                    ld4s<T>(&s_cf[w][k][j][4 * (comp ^ ((j >> 1) & 3))], C);
                    T t = B[0] * C[0];
                    t = fma(B[1], C[1], t);
                    t = fma(B[2], C[2], t);
                    t = fma(B[3], C[3], t);
                    sum[k] += t;
                }
            }
            for (int k = 0; k < 4; ++k) acc[32 * (4 * b + k)] += sum[k];
            __syncwarp();
        }
        __syncthreads();   // the test functions are replaced
    }
    if (MODE == FULL) {
        for (int s = 4 * NB * w; s < 4 * NB * (w + 1); ++s) K[(int64_t)sl * 1024 + lane * 32 + s] = (double)acc[32 * s];
        return;
    }
    __syncthreads();
    if (MODE == BSR) {
        constexpr int NP = 64 / JWPB;   // corner pairs per warp: pair (m / 8, m % 8), m = NP w ...
        int64_t* s_pos = reinterpret_cast<int64_t*>(&s_cf[w][0][0][0]);   // (the points are done)
        const unsigned hanging = __ballot_sync(0xffffffffu, lane < 8 && !plain_corner(A, my_id)) & 0xffu;
        const int pm = NP * w + (lane & (NP - 1)), pa = pm >> 3, pb = pm & 7;
        const int32_t ida = __shfl_sync(0xffffffffu, my_id, pa), idb = __shfl_sync(0xffffffffu, my_id, pb);
        if (lane < NP) s_pos[lane] = (hanging >> pa | hanging >> pb) & 1u ? -1 : bsr_find(A.bptr, A.bidx, ida, idb);
        __syncwarp();
        bsr_add_blocks<NP>(s_pos, [&](int m, int j) {
            const int q = NP * w + m;
            return s_acc[4 * (q & 7) + (j & 3)][4 * (q >> 3) + (j >> 2)];
        }, lane, K);
        if (hanging)
            for (int m = NP * w; m < NP * (w + 1); ++m) {
                const int ha = m >> 3, hb = m & 7;
                if (!((hanging >> ha | hanging >> hb) & 1u)) continue;
                const int32_t ia = __shfl_sync(0xffffffffu, my_id, ha), ib = __shfl_sync(0xffffffffu, my_id, hb);
                bsr_add_hanging(A, ia, ib, [&](int j) { return s_acc[4 * hb + (j & 3)][4 * ha + (j >> 2)]; }, lane, K);
            }
    } else if (w == 0) {
        // lane (a, comp) holds row comp of corner a's own block in columns 4a .. 4a+3
        double blk[16];
        for (int i = 0; i < 4; ++i)
            for (int k = 0; k < 4; ++k) blk[i * 4 + k] = (double)s_acc[4 * a + k][4 * a + i];
        const int32_t id = __shfl_sync(0xffffffffu, my_id, a);
        if (comp == 0) add_diag(A, id, blk, D);
    }
}

template <int MODE>
__global__ void __launch_bounds__(128) jac_nitsche(Args A, const int32_t* __restrict__ el,
                                                   const double* __restrict__ xr, const double* __restrict__ nr,
                                                   const double* __restrict__ wr, const double* __restrict__ taub,
                                                   int64_t n, const int32_t* __restrict__ slot, double* __restrict__ K,
                                                   double* __restrict__ D) {
    typedef float T;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t e = el[i];
    const int32_t sl = MODE == FULL ? slot[e] : 0;
    if (sl < 0) return;
    NitschePoint<T, T> V;
    nitsche_fields<T, T, false>(A, e, i, xr + 3 * i, nr + 3 * i, V);
    const T w = (T)wr[i];
    const T tauB = (T)(A.Cb * (double)V.mu * taub[i]);
    for (int b = 0; b < 8; ++b) {
        for (int k = 0; k < 4; ++k) {
            // tangent point data of the seed (corner b, component k)
            NitschePoint<Dual<T>, T> P;
            P.g = V.g;
            P.mu = V.mu;
            P.rho = V.rho;
            P.B = V.B;
            for (int c = 0; c < 8; ++c) P.ids[c] = V.ids[c];
            for (int j = 0; j < 3; ++j) P.nn[j] = V.nn[j];
            const T th = (T)A.theta, phb = V.B.phi[b];
            P.p = {V.p, k == 3 ? phb : T(0)};
            for (int kk = 0; kk < 3; ++kk) {
                P.us[kk] = {V.us[kk], kk == k ? th * phb : T(0)};
                P.d[kk] = {V.d[kk], kk == k ? th * phb : T(0)};
                for (int j = 0; j < 3; ++j)
                    P.Gu[kk][j] = {V.Gu[kk][j], kk == k ? th * V.B.dphi[b][j] : T(0)};   // reference; scaled below
            }
            // finish_nitsche scales Gu by g: undo for the values (already physical)
            for (int kk = 0; kk < 3; ++kk)
                for (int j = 0; j < 3; ++j) P.Gu[kk][j].v = V.Gu[kk][j] / V.g;
            finish_nitsche(A, P);
            P.inflow = V.inflow;
            if (MODE == FULL) {
                for (int c = 0; c < 8; ++c) {
                    Dual<T> t[4];
                    nitsche_rows<Dual<T>, T>(A, P, c, tauB, t);
                    for (int r = 0; r < 4; ++r)
                        atomicAdd(K + (int64_t)sl * 1024 + (c * 4 + r) * 32 + b * 4 + k, (double)(w * t[r].d));
                }
            } else {
                Dual<T> t[4];
                nitsche_rows<Dual<T>, T>(A, P, b, tauB, t);
                double blk[16];
                for (int q = 0; q < 16; ++q) blk[q] = 0.0;
                for (int r = 0; r < 4; ++r) blk[r * 4 + k] = (double)(w * t[r].d);
                add_diag(A, P.ids[b], blk, D);
            }
        }
    }
}

// ------------------------------------------------------------------------------------------
// Float64: a warp per element part, lane = column (corner b, component k) of k_e.  The FP64 pipe is the
// bound (see Const64), so what does not depend on the column is formed once per point, with a lane per
// point (fields by Horner steps, the value part of the pointwise terms: about 165 FP64 instructions for 32
// points), and kept in shared memory; the columns then differentiate around those values with a seed
// whose zeros are spelled out (100 per point) and add their 32 test moments in registers (80).  The
// seed-by-seed dual numbers of the float32 kernels below took about 900 per point.
//   jac_out64   four Out elements per warp: 4 x 8 Gauss points at once, then the elements in turn
//   jac_cut64   a block of four warps per Intercepted element, 32 sub-cell points per warp at a time
//   jac_surf64  a warp per element hosting surface points: no atomics between its points
// 8,192 of 33.7 k elements (a ninth of them Intercepted, 288 points each): 35.8 -> 4.5 ms.
// ------------------------------------------------------------------------------------------
enum { JX = 0, JU = 3, JG = 6, JUP = 15, JGU = 18, JC = 21, JA = 24, JQ = 27, JDIV = 31, JS = 32, JS2 = 33, JNRR = 34,
       JNRG = 35, JNRM = 36, JMP = 37, JWM = 38, JN = 46 };
constexpr int JSTR = 33;             // point stride of a stored quantity
constexpr int JWARP = JN * JSTR;     // doubles of a warp's point area

// value columns of element e as Hadamard coefficients, [column][8] (columns 7-9: force)
__device__ __forceinline__ void jac_columns64(const Args& A, int32_t e, double* s_col, int t0, int nt) {
    for (int t = t0; t < 96; t += nt) {
        const int col = t >> 3, c = t & 7;
        const int64_t id = A.conn[8 * (int64_t)e + c];
        double x = 0.0;
        if (col < 7) x = __ldg((const double*)A.ndv + 8 * id + col);
        else if (col < 10 && A.ndf) x = __ldg((const double*)A.ndf + 4 * id + col - 7);
        s_col[t] = hadamard_fwd(x, c);
    }
}

// the column-independent quantities of a point (8-fold fields), stored at s[.. * JSTR]; w: its weight / 64
__device__ __forceinline__ void jac_point64(const Args& A, const Const64& C, const double* s_col, double x, double y, double z,
                                            double w, double* s) {
    auto value = [&](int col) {
        const double* a = s_col + 8 * col;
        const double b0 = fma(x, a[1], a[0]), b1 = fma(x, a[3], a[2]), b2 = fma(x, a[5], a[4]), b3 = fma(x, a[7], a[6]);
        return fma(z, fma(y, b3, b2), fma(y, b1, b0));
    };
    double u[3], G[3][3], p, gp[3], H[3], m[3][3], none[3];
    auto all = [&](int col, double& v, double g[3], double d2[3]) {   // as in the Intercepted J v kernel
        const double* a = s_col + 8 * col;
        const double b0 = fma(x, a[1], a[0]), b1 = fma(x, a[3], a[2]), b2 = fma(x, a[5], a[4]), b3 = fma(x, a[7], a[6]);
        const double c1 = fma(y, b3, b2), j = fma(y, a[7], a[5]);
        v = fma(z, c1, fma(y, b1, b0));
        g[2] = c1;
        g[1] = fma(z, b3, b1);
        g[0] = fma(z, j, fma(y, a[3], a[1]));
        d2[0] = fma(z, a[7], a[3]);
        d2[1] = j;
        d2[2] = b3;
    };
    for (int i = 0; i < 3; ++i) all(i, u[i], G[i], m[i]);
    H[0] = m[1][0] + m[2][1];
    H[1] = m[0][0] + m[2][2];
    H[2] = m[0][1] + m[1][2];
    all(3, p, gp, none);
    double Gg[3][3], rM[3], up[3], GU[3];
    for (int i = 0; i < 3; ++i) {
        for (int j = 0; j < 3; ++j) Gg[i][j] = C.g8 * G[i][j];
        double acc = fma(Gg[i][2], u[2], fma(Gg[i][1], u[1], fma(Gg[i][0], u[0], value(4 + i))));
        if (A.ndf) acc -= value(7 + i);
        rM[i] = fma(C.rho, acc, fma(-C.mug2, H[i], C.g * gp[i]));
    }
    const double arg = fma(C.g264, fma(u[2], u[2], fma(u[1], u[1], u[0] * u[0])), C.K);
    const double r = rsqrt(arg), tC = (arg * r) * C.i3g2;
    for (int i = 0; i < 3; ++i) up[i] = -r * rM[i];
    const double q = C.g264 * fma(up[2], up[2], fma(up[1], up[1], up[0] * up[0]));
    const double sb = q > tiny<double>() ? rsqrt(q) : 0.0;
    const double rg = (r * r) * C.g264;
    s[JX * JSTR] = x;
    s[(JX + 1) * JSTR] = y;
    s[(JX + 2) * JSTR] = z;
    for (int i = 0; i < 3; ++i) {
        GU[i] = fma(Gg[i][2], up[2], fma(Gg[i][1], up[1], Gg[i][0] * up[0]));
        s[(JU + i) * JSTR] = u[i];
        for (int j = 0; j < 3; ++j) s[(JG + 3 * i + j) * JSTR] = Gg[i][j];
        s[(JUP + i) * JSTR] = up[i];
        s[(JGU + i) * JSTR] = GU[i];
        s[(JC + i) * JSTR] = fma(sb, GU[i], -C.irho * up[i]);
        s[(JA + i) * JSTR] = C.kap8 * up[i];
        s[(JQ + i) * JSTR] = rg * u[i];
    }
    s[(JQ + 3) * JSTR] = 0.0;
    s[JDIV * JSTR] = G[0][0] + G[1][1] + G[2][2];
    s[JS * JSTR] = sb;
    s[JS2 * JSTR] = (sb * sb) * C.g264;
    s[JNRR * JSTR] = -r * C.rho;
    s[JNRG * JSTR] = -r * C.g;
    s[JNRM * JSTR] = r * C.mug2;
    s[JMP * JSTR] = C.kap * (tC * C.rhog);
    const double wx = w * x, wy = w * y, wxy = wx * y;
    const double wm[8] = {w, wx, wy, wxy, w * z, wx * z, wy * z, wxy * z};
    for (int t = 0; t < 8; ++t) s[(JWM + t) * JSTR] = wm[t];
}

// 8-fold basis function of corner b at (x, y, z): phi, reference gradient d, mixed second derivatives (xy, xz, yz)
__device__ __forceinline__ void jac_seed64(int b, double x, double y, double z, double& phi, double d[3], double m[3]) {
    const double fx = (b & 1) ? 1.0 + x : 1.0 - x, fy = (b & 2) ? 1.0 + y : 1.0 - y, fz = (b & 4) ? 1.0 + z : 1.0 - z;
    const double fyz = fy * fz, fxz = fx * fz, fxy = fx * fy;
    phi = fx * fyz;
    d[0] = (b & 1) ? fyz : -fyz;
    d[1] = (b & 2) ? fxz : -fxz;
    d[2] = (b & 4) ? fxy : -fxy;
    m[0] = (((b >> 1) ^ b) & 1) ? -fz : fz;
    m[1] = (((b >> 2) ^ b) & 1) ? -fy : fy;
    m[2] = (((b >> 2) ^ (b >> 1)) & 1) ? -fx : fx;
}

// moments of one column's coefficients: f, s of component i with weighted monomials m
__device__ __forceinline__ void jac_moments64(const double m[8], int i, double f, double sx, double sy, double sz, double M[32]) {
    auto add = [&](int S, double a, double v) { M[4 * S + i] = fma(a, v, M[4 * S + i]); };
    add(0, m[0], f);
    add(1, m[1], f); add(1, m[0], sx);
    add(2, m[2], f); add(2, m[0], sy);
    add(3, m[3], f); add(3, m[2], sx); add(3, m[1], sy);
    add(4, m[4], f); add(4, m[0], sz);
    add(5, m[5], f); add(5, m[4], sx); add(5, m[1], sz);
    add(6, m[6], f); add(6, m[4], sy); add(6, m[2], sz);
    add(7, m[7], f); add(7, m[6], sx); add(7, m[5], sy); add(7, m[3], sz);
}

// Column (b, k) at the stored point s, theta left out (the finished column is scaled): the derivative for
// the seed du_k = phi, or dp = phi.  DIAG: adds the four rows of corner b itself to M[0 .. 4), else the
// 32 test moments.
template <bool DIAGM>
__device__ __forceinline__ void jac_column64(const Const64& C, double ratio, const double* s, int b, int k, double* M) {
    auto ld = [&](int f) { return s[f * JSTR]; };
    double phi, d[3], m[3];
    jac_seed64(b, ld(JX), ld(JX + 1), ld(JX + 2), phi, d, m);
    const bool isp = k == 3;
    const double X = fma(C.g8, fma(d[2], ld(JU + 2), fma(d[1], ld(JU + 1), d[0] * ld(JU))), ratio * phi);
    const double phiv = isp ? 0.0 : phi;
    const int kk = isp ? 0 : k;
    // grad p, or the mixed derivatives of u_k that enter (grad div u)_i, i != k
    const double v[3] = {k == 1 ? m[0] : k == 2 ? m[1] : isp ? d[0] : 0.0, k == 0 ? m[0] : k == 2 ? m[2] : isp ? d[1] : 0.0,
                         k == 0 ? m[1] : k == 1 ? m[2] : isp ? d[2] : 0.0};
    const double coef = s[(isp ? JNRG : JNRM) * JSTR], h = s[(JQ + k) * JSTR] * phi, nrr = ld(JNRR);
    double dacc[3], dup[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        dacc[i] = fma(s[(JG + 3 * i + kk) * JSTR], phiv, i == k ? X : 0.0);
        dup[i] = fma(nrr, dacc[i], fma(-h, ld(JUP + i), coef * v[i]));
    }
    const double hs = ld(JS2) * fma(ld(JUP + 2), dup[2], fma(ld(JUP + 1), dup[1], ld(JUP) * dup[0]));
    const double t2 = C.g8 * fma(d[2], ld(JUP + 2), fma(d[1], ld(JUP + 1), d[0] * ld(JUP)));
    const double ddiv = k == 0 ? d[0] : k == 1 ? d[1] : k == 2 ? d[2] : 0.0;
    const double kphi = C.kap * phi;
    const double dP = fma(-ld(JMP), fma(h, ld(JDIV), ddiv), isp ? kphi : 0.0);
    double F[3], dc[3], dA[3], Hh[3], mj[3], tk[3];
    const double sb = ld(JS);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double dGU = fma(ld(JG + 3 * i), dup[0], fma(ld(JG + 3 * i + 1), dup[1], fma(ld(JG + 3 * i + 2), dup[2], i == k ? t2 : 0.0)));
        F[i] = fma(C.rho, dacc[i], dGU);
        const double dw = -C.irho * dup[i];
        dc[i] = fma(sb, fma(-hs, ld(JGU + i), dGU), dw);
        dA[i] = C.kap8 * dup[i];
        Hh[i] = C.kap * dw;
        mj[i] = C.mgk * d[i];
        tk[i] = fma(-ld(JA + i), phi, mj[i]);
    }
    double m8[8], ph4 = 0.0, g4[3] = {0.0, 0.0, 0.0};
    if (DIAGM) {
        ph4 = ld(JWM) * phi;
        for (int j = 0; j < 3; ++j) g4[j] = ld(JWM) * d[j];
    } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) m8[t] = ld(JWM + t);
    }
    auto put = [&](int i, double f, double sx, double sy, double sz) {
        if (DIAGM) M[i] = fma(ph4, f, fma(g4[0], sx, fma(g4[1], sy, fma(g4[2], sz, M[i]))));
        else jac_moments64(m8, i, f, sx, sy, sz, M);
    };
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double S[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            // mu (dG_ij + dG_ji) - u'_i du_j, and the pressure on the diagonal
            double e = j == k ? tk[i] : i == k ? mj[j] : 0.0;
            if (i == j) e = (i == k ? e + mj[i] : e) - dP;
            S[j] = fma(-dA[i], ld(JU + j), fma(dc[i], ld(JA + j), fma(ld(JC + i), dA[j], e)));
        }
        put(i, F[i], S[0], S[1], S[2]);
    }
    put(3, C.g * ddiv, Hh[0], Hh[1], Hh[2]);
}

// test moments -> rows of the 8 corners (one column per lane), velocity columns times theta
__device__ __forceinline__ void jac_rows64(const Args& A, int k, double M[32]) {
#pragma unroll
    for (int ax = 0; ax < 3; ++ax)
#pragma unroll
        for (int t = 0; t < 8; ++t)
            if (!(t & (1 << ax)))
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const double lo = M[4 * t + i], hi = M[4 * (t | (1 << ax)) + i];
                    M[4 * t + i] = lo - hi;
                    M[4 * (t | (1 << ax)) + i] = lo + hi;
                }
    if (!A.theta1 && k < 3)
        for (int t = 0; t < 32; ++t) M[t] *= A.theta;
}

// the warp's finished columns: FULL to K (add: onto what is there), BSR into the assembled blocks through
// M_e (one search of the row per corner pair, not per entry), DIAG (M[0 .. 4): corner b's own rows) to D
template <int MODE>
__device__ __forceinline__ void jac_store64(const Args& A, int32_t e, int64_t sl, double* M, int lane, double* __restrict__ K,
                                            double* __restrict__ D, bool add) {
    const int b = lane >> 2, k = lane & 3;
    if (MODE == FULL) {
        double* o = K + sl * 1024 + lane;
#pragma unroll
        for (int r = 0; r < 32; ++r) o[32 * r] = add ? o[32 * r] + M[r] : M[r];
        return;
    }
    int32_t nb[4];
    double wb;
    const int cb = corner_nodes(A, A.conn[8 * (int64_t)e + b], nb, wb);
    if (MODE == DIAG) {
        for (int p = 0; p < cb; ++p)
            for (int i = 0; i < 4; ++i) atomicAdd(D + 16 * (int64_t)nb[p] + 4 * i + k, wb * wb * M[i]);
        return;
    }
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        int32_t na[4];
        double wa;
        const int ca = corner_nodes(A, A.conn[8 * (int64_t)e + a], na, wa);
        for (int p = 0; p < ca; ++p)
            for (int q = 0; q < cb; ++q) {
                const int64_t pos = bsr_find(A.bptr, A.bidx, na[p], nb[q]);
                if (pos < 0) continue;
                double* o = K + 16 * pos + k;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (M[4 * a + i] != 0.0) atomicAdd(o + 4 * i, wa * wb * M[4 * a + i]);
            }
    }
}

template <int MODE> struct JacAcc { static constexpr int n = MODE == DIAG ? 4 : 32; };

constexpr int J64W = 4;   // warps per block
inline size_t jac64_smem() { return (size_t)J64W * (JWARP + 4 * 96) * sizeof(double); }

// list: the Out elements, or (FULL) the requested elements, of which this kernel takes the Out ones
template <int MODE>
__global__ void __launch_bounds__(32 * J64W, 2) jac_out64(Args A, const int32_t* __restrict__ list, int64_t n,
                                                         const int8_t* __restrict__ marker, const int32_t* __restrict__ slot,
                                                         double* __restrict__ K, double* __restrict__ D) {
    extern __shared__ __align__(16) double sm[];
    const int lane = threadIdx.x & 31, le = lane >> 3, w = threadIdx.x >> 5;
    double* s = sm + w * (JWARP + 4 * 96);
    double* s_col = s + JWARP;
    const int64_t i0 = ((int64_t)blockIdx.x * J64W + w) * 4;
    if (i0 >= n) return;
    auto takes = [&](int64_t i) {   // element of position i if it is ours, else -1
        if (i >= n) return -1;
        const int32_t e = list[i];
        return MODE != FULL || (marker[e] == 0 && slot[e] == (int32_t)i) ? e : -1;
    };
    const int32_t mine = takes(i0 + le);
    if (!__any_sync(0xffffffffu, mine >= 0)) return;
    for (int q = 0; q < 4; ++q) {
        const int32_t e = __shfl_sync(0xffffffffu, mine, 8 * q);
        if (e >= 0) jac_columns64(A, e, s_col + 96 * q, lane, 32);
    }
    __syncwarp();
    if (mine >= 0) {
        const int lv = A.lev[mine];
        const Const64 C(A, Phys<double>(A, prob_of(A, mine)), lv, A.lc[lv][0], A.lc[lv][1]);
        const double gam = kGauss;
        jac_point64(A, C, s_col + 96 * le, (lane & 1) ? gam : -gam, (lane & 2) ? gam : -gam, (lane & 4) ? gam : -gam,
                    A.lc[lv][6], s + lane);
    }
    __syncwarp();
    const int b = lane >> 2, k = lane & 3;
    for (int q = 0; q < 4; ++q) {
        const int32_t e = __shfl_sync(0xffffffffu, mine, 8 * q);
        if (e < 0) continue;
        const int lv = A.lev[e];
        const Const64 C(A, Phys<double>(A, prob_of(A, e)), lv, A.lc[lv][0], A.lc[lv][1]);
        double M[JacAcc<MODE>::n];
#pragma unroll
        for (int t = 0; t < JacAcc<MODE>::n; ++t) M[t] = 0.0;
        for (int j = 0; j < 8; ++j) jac_column64<MODE == DIAG>(C, A.c0th, s + 8 * q + j, b, k, M);
        if constexpr (MODE == DIAG) {
            if (!A.theta1 && k < 3)
                for (int t = 0; t < 4; ++t) M[t] *= A.theta;
        } else {
            jac_rows64(A, k, M);
        }
        jac_store64<MODE>(A, e, i0 + q, M, lane, K, D, false);
    }
}

template <int MODE>
__global__ void __launch_bounds__(32 * J64W, 2) jac_cut64(Args A, const int32_t* __restrict__ list, const int64_t* __restrict__ off,
                                                         const double* __restrict__ pts, const int32_t* __restrict__ order,
                                                         const int32_t* __restrict__ slot, double* __restrict__ K,
                                                         double* __restrict__ D) {
    extern __shared__ __align__(16) double sm[];
    constexpr int NA = JacAcc<MODE>::n;
    static_assert(32 * 32 <= JWARP, "the parts' sums take the point areas");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t idx = order[blockIdx.x];
    const int32_t e = list[idx];
    const int64_t sl = MODE == FULL ? slot[e] : 0;
    if (sl < 0) return;
    double *s = sm + w * JWARP, *s_col = sm + J64W * JWARP;
    jac_columns64(A, e, s_col, threadIdx.x, 32 * J64W);
    const int lv = A.lev[e];
    const Const64 C(A, Phys<double>(A, prob_of(A, e)), lv, A.lc[lv][0], A.lc[lv][1]);
    const int64_t q0 = off[idx], q1 = off[idx + 1];
    const int b = lane >> 2, k = lane & 3;
    double M[NA];
#pragma unroll
    for (int t = 0; t < NA; ++t) M[t] = 0.0;
    __syncthreads();
    for (int64_t base = q0 + 32 * w; base < q1; base += 32 * J64W) {
        const int cnt = (int)min((int64_t)32, q1 - base);
        if (lane < cnt) {
            double pt[4];
            load_pt<double>(pts, base + lane, pt);
            jac_point64(A, C, s_col, pt[0], pt[1], pt[2], pt[3] * A.lc[lv][6], s + lane);
        }
        __syncwarp();
        for (int j = 0; j < cnt; ++j) jac_column64<MODE == DIAG>(C, A.c0th, s + j, b, k, M);
        __syncwarp();
    }
    // the warps' sums in order (the point areas are free)
#pragma unroll
    for (int t = 0; t < NA; ++t) s[32 * t + lane] = M[t];
    __syncthreads();
    if (w > 0) return;
    for (int p = 1; p < J64W && q0 + 32 * p < q1; ++p)
#pragma unroll
        for (int t = 0; t < NA; ++t) M[t] += sm[p * JWARP + 32 * t + lane];
    if constexpr (MODE == DIAG) {
        if (!A.theta1 && k < 3)
            for (int t = 0; t < 4; ++t) M[t] *= A.theta;
    } else {
        jac_rows64(A, k, M);
    }
    jac_store64<MODE>(A, e, sl, M, lane, K, D, false);
}

// Surface terms (rows of nitsche_rows) of a host element: points [pq[i], pq[i + 1]) of element pe[i]; runs
// after the volume kernels (FULL: adds to their k_e)
template <int MODE>
__global__ void __launch_bounds__(128) jac_surf64(Args A, const int32_t* __restrict__ pe, const int64_t* __restrict__ pq,
                                                  const double* __restrict__ xr, const double* __restrict__ nr,
                                                  const double* __restrict__ wr, const double* __restrict__ taub, int64_t n,
                                                  const int32_t* __restrict__ slot, double* __restrict__ K, double* __restrict__ D) {
    __shared__ double s_col[4][96], s_pt[4][8][JSTR];   // point: velocity jump (0-2), u.n / |rho, inflow| (3), weight (4), tau_B (5)
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * 4 + w;
    if (i >= n) return;
    const int32_t e = pe[i];
    const int64_t sl = MODE == FULL ? slot[e] : 0;
    if (sl < 0) return;
    jac_columns64(A, e, s_col[w], lane, 32);
    const Phys<double> P(A, prob_of(A, e));
    const double g = A.lc[A.lev[e]][0], mg = P.mu * g;
    const int b = lane >> 2, k = lane & 3;
    double M[JacAcc<MODE>::n];
#pragma unroll
    for (int t = 0; t < JacAcc<MODE>::n; ++t) M[t] = 0.0;
    __syncwarp();
    const int64_t q1 = pq[i + 1];
    for (int64_t base = pq[i]; base < q1; base += 32) {
        const int cnt = (int)min((int64_t)32, q1 - base);
        if (lane < cnt) {
            const int64_t q = base + lane;
            const double *x = xr + 3 * q, *nn = nr + 3 * q, *gq = point_g(A, q);
            double un = 0.0;
            for (int j = 0; j < 3; ++j) {
                const double* a = s_col[w] + 8 * j;
                const double b0 = fma(x[0], a[1], a[0]), b1 = fma(x[0], a[3], a[2]), b2 = fma(x[0], a[5], a[4]), b3 = fma(x[0], a[7], a[6]);
                const double u = 0.125 * fma(x[2], fma(x[1], b3, b2), fma(x[1], b1, b0));
                un = fma(u, nn[j], un);
                s_pt[w][j][lane] = u - gq[j];
            }
            s_pt[w][3][lane] = un < 0.0 ? P.rho * un : 0.0;
            s_pt[w][4][lane] = wr[q] * 0.015625;   // 8-fold seed and test functions
            s_pt[w][5][lane] = A.Cb * P.mu * taub[q];
        }
        __syncwarp();
        for (int j = 0; j < cnt; ++j) {
            const int64_t q = base + j;
            const double x = xr[3 * q], y = xr[3 * q + 1], z = xr[3 * q + 2];
            const double nn[3] = {nr[3 * q], nr[3 * q + 1], nr[3 * q + 2]};
            double phi, d[3], m[3];
            jac_seed64(b, x, y, z, phi, d, m);
            const double wq = s_pt[w][4][j];
            const bool isp = k == 3;
            const double nk = k == 0 ? nn[0] : k == 1 ? nn[1] : k == 2 ? nn[2] : 0.0;
            const double ph = isp ? 0.0 : phi;
            const double dn = fma(d[2], nn[2], fma(d[1], nn[1], d[0] * nn[0]));
            const double run = s_pt[w][3][j];                                     // rho u.n where u.n < 0
            const double rin = run < 0.0 ? P.rho : 0.0;
            const double diag = fma(s_pt[w][5][j] - run, ph, isp ? 0.0 : -mg * dn);   // coefficient on i = k
            double F[3];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                // -tr_i + tau_B d_i - [u.n < 0] rho ((u.n)' (u - g)_i + u.n d_i)
                double f = isp ? phi * nn[r] : -mg * (d[r] * nk);
                f = fma(-(rin * nk) * ph, s_pt[w][r][j], f);
                F[r] = wq * (r == k ? f + diag : f);
            }
            const double wmg = -(wq * mg) * ph, wn = -wq * (nk * ph);
            if (MODE == DIAG) {
                for (int r = 0; r < 3; ++r) {
                    double f = phi * F[r];
                    // S_rj = -mu (n_j d_r + n_r d_j) in reference gradients
                    f = fma(wmg, (r == k ? dn : 0.0) + nn[r] * (k == 0 ? d[0] : k == 1 ? d[1] : d[2]), f);
                    M[r] += f;
                }
                M[3] = fma(phi, wn, M[3]);
            } else {
                const double xy = x * y;
                const double m8[8] = {1.0, x, y, xy, z, x * z, y * z, xy * z};
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    double S[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) S[c] = wmg * ((r == k ? nn[c] : 0.0) + (c == k ? nn[r] : 0.0));
                    jac_moments64(m8, r, F[r], S[0], S[1], S[2], M);
                }
                jac_moments64(m8, 3, wn, 0.0, 0.0, 0.0, M);
            }
        }
        __syncwarp();
    }
    if constexpr (MODE == DIAG) {
        if (!A.theta1 && k < 3)
            for (int t = 0; t < 4; ++t) M[t] *= A.theta;
    } else {
        jac_rows64(A, k, M);
    }
    jac_store64<MODE>(A, e, sl, M, lane, K, D, true);
}

// Element Jacobians asked for whole (FULL): the Intercepted elements' kernel on a side stream beside the Out
// elements', forked after the node rows and joined before the surface terms are added; every k_e has one writer,
// so nothing depends on the order.  Each kernel alone leaves the last of its few waves of blocks half empty
// (33.7 k elements, float64: 4.47 -> 4.14 ms).  Not for the modes that add with atomics, whose order a mixed
// solve can turn into other last digits (an assembly of 43.6 k elements would gain 5 %), and not under
// capture, where a side stream would stay in the capture it was forked in.
struct JacFork {
    cudaStream_t s, cut;
    cudaEvent_t* ev = nullptr;
    JacFork(const Mesh& m, cudaStream_t stream, bool full) : s(stream), cut(stream) {
        Mesh& mm = const_cast<Mesh&>(m);
        cudaStreamCaptureStatus st = cudaStreamCaptureStatusActive;
        if (!full || !m.concurrent || cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone ||
            side_streams(mm)) return;
        cut = (cudaStream_t)m.side[0];
        ev = (cudaEvent_t*)mm.fork_ev;
        cudaEventRecord(ev[0], s);
        cudaStreamWaitEvent(cut, ev[0], 0);
    }
    void join() {
        if (!ev) return;
        cudaEventRecord(ev[1], cut);
        cudaStreamWaitEvent(s, ev[1], 0);
    }
};

// every float64 kernel; FULL: elems (n of them) the requested elements and slot their positions
template <int MODE>
void launch_jac64(const Mesh& m, Args A, const int32_t* elems, int64_t n, const int32_t* slot, double* K, double* D, cudaStream_t s) {
    const int64_t next = m.n_nodes() + m.n_hang();
    double* ndv = node_workspace<double>(m, nullptr);
    A.ndv = ndv;
    A.ndt = ndv + 8 * next;
    A.ndf = A.F ? ndv + 16 * next : nullptr;
    if (next > 0) launch_node_prep<double, false>(A, ndv, ndv + 8 * next, (double*)A.ndf, s);
    const int64_t no = MODE == FULL ? n : (int64_t)m.out_list.size(), nc = (int64_t)m.cut_list.size(), np = (int64_t)m.pen_elem.size();
    const size_t smem = jac64_smem();
    // (set on every call: the attribute belongs to the current device)
    cudaFuncSetAttribute(jac_out64<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(jac_cut64<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    JacFork f(m, s, MODE == FULL);
    // the Intercepted elements first, as their blocks are the long ones
    if (nc > 0)
        jac_cut64<MODE><<<(unsigned)nc, 32 * J64W, smem, f.cut>>>(A, m.d.cut_list, m.d.cut_off, m.d.cut_pts, m.d.cut_order, slot, K, D);
    if (no > 0)
        jac_out64<MODE><<<(unsigned)((no + 4 * J64W - 1) / (4 * J64W)), 32 * J64W, smem, s>>>(A, MODE == FULL ? elems : m.d.out_list, no,
                                                                                          m.d.marker, slot, K, D);
    f.join();
    if (np > 0)
        jac_surf64<MODE><<<(unsigned)((np + 3) / 4), 128, 0, s>>>(A, m.d.pen_elem, m.d.pen_q, m.d.sq_x, m.d.sq_n, m.d.sq_w, m.d.sq_taub,
                                                                 np, slot, K, D);
}

// rows of prescribed components become identity rows
__global__ void jac_strong_rows(int64_t nn, const uint8_t* __restrict__ flag, const uint8_t* __restrict__ umask,
                                double* __restrict__ D) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= nn) return;
    uint8_t mask = umask ? umask[n] : (uint8_t)(flag[n] & 15);
    if (flag[n] & 16) mask = 15;
    for (int k = 0; k < 4; ++k)
        if ((mask >> k) & 1)
            for (int j = 0; j < 4; ++j) D[16 * n + 4 * k + j] = j == k ? 1.0 : 0.0;
}

// invert every 4x4 block (Gauss-Jordan, partial pivoting, float64); a singular block -> identity
__global__ void bj_invert(int64_t nn, const double* __restrict__ D, double* __restrict__ Dinv) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= nn) return;
    double a[4][8];
    double scale = 0.0;
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) {
            a[i][j] = D[16 * n + 4 * i + j];
            a[i][4 + j] = i == j ? 1.0 : 0.0;
            scale = fmax(scale, fabs(a[i][j]));
        }
    bool ok = scale > 0.0;
    for (int col = 0; col < 4 && ok; ++col) {
        int piv = col;
        for (int r = col + 1; r < 4; ++r)
            if (fabs(a[r][col]) > fabs(a[piv][col])) piv = r;
        if (!(fabs(a[piv][col]) > 1e-14 * scale)) { ok = false; break; }
        if (piv != col)
            for (int j = 0; j < 8; ++j) { double t = a[col][j]; a[col][j] = a[piv][j]; a[piv][j] = t; }
        const double inv = 1.0 / a[col][col];
        for (int j = 0; j < 8; ++j) a[col][j] *= inv;
        for (int r = 0; r < 4; ++r) {
            if (r == col) continue;
            const double f = a[r][col];
            if (f != 0.0)
                for (int j = 0; j < 8; ++j) a[r][j] -= f * a[col][j];
        }
    }
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) Dinv[16 * n + 4 * i + j] = ok ? a[i][4 + j] : (i == j ? 1.0 : 0.0);
}

// y_n = Dinv_n x_n
__global__ void bj_apply(int64_t nn, const double* __restrict__ Dinv, const double* __restrict__ x,
                         double* __restrict__ y) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= nn) return;
    const double* M = Dinv + 16 * n;
    double xv[4] = {x[4 * n], x[4 * n + 1], x[4 * n + 2], x[4 * n + 3]};
    for (int i = 0; i < 4; ++i) y[4 * n + i] = M[4 * i] * xv[0] + M[4 * i + 1] * xv[1] + M[4 * i + 2] * xv[2] + M[4 * i + 3] * xv[3];
}

__global__ void fill_slots(int64_t n, const int32_t* __restrict__ list, int32_t* __restrict__ slot) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) slot[list[i]] = (int32_t)i;
}

template <int MODE>
void launch_jac(const Mesh& m, Args A, const int32_t* slot, double* K, double* D, cudaStream_t s) {
    const int64_t next = m.n_nodes() + m.n_hang();
    float* ndv = node_workspace<float>(m, nullptr);
    A.ndv = ndv;
    A.ndt = ndv + 8 * next;
    A.ndf = A.F ? ndv + 16 * next : nullptr;
    if (next > 0)
        launch_node_prep<float, false>(A, ndv, ndv + 8 * next, (float*)A.ndf, s);
    const int64_t no = (int64_t)m.out_list.size(), nc = (int64_t)m.cut_list.size(), ns = (int64_t)m.sq.size() / 10;
    constexpr int EPB = kOutEpb;
    JacFork f(m, s, MODE == FULL);
    if (no > 0) jac_out<MODE><<<(unsigned)((no + EPB - 1) / EPB), 8 * EPB, 0, s>>>(A, m.d.out_list, no, slot, K, D);
    if (nc > 0)
        jac_cut<MODE><<<(unsigned)nc, 32 * JWPB, 0, f.cut>>>(A, m.d.cut_list, m.d.cut_off, m.d.cut_pts_f, m.d.cut_order, slot, K, D);
    f.join();
    if (ns > 0)
        jac_nitsche<MODE><<<(unsigned)((ns + 31) / 32), 32, 0, s>>>(A, m.d.sq_elem, m.d.sq_x, m.d.sq_n, m.d.sq_w, m.d.sq_taub, ns,
                                                                    slot, K, D);
}

// k_e of the surface terms (one per host element, slot order) added to the assembled matrix
__global__ void scatter_kmat(Args A, const int32_t* __restrict__ list, int64_t n, const double* __restrict__ Ks,
                             double* __restrict__ val) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // (element, row, column block)
    if (t >= n * 256) return;
    const int64_t s = t >> 8;
    const int row = (int)((t >> 3) & 31), b = (int)(t & 7);
    const int32_t e = list[s];
    const int32_t ida = A.conn[8 * (int64_t)e + (row >> 2)], idb = A.conn[8 * (int64_t)e + b];
    const int comp = row & 3;
    bsr_add<4>(A, ida, idb, Ks + s * 1024 + row * 32 + 4 * b, [=](int j) { return 4 * comp + j; }, val);
}

// rows of prescribed components become identity rows of the assembled matrix; eight threads per node
// over its blocks
__global__ void bsr_strong_rows(int64_t nn, const int64_t* __restrict__ ptr, const int32_t* __restrict__ idx,
                                const uint8_t* __restrict__ flag, const uint8_t* __restrict__ umask, double* __restrict__ val) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, n = t >> 3;
    if (n >= nn) return;
    uint8_t mask = umask ? umask[n] : (uint8_t)(flag[n] & 15);
    if (flag[n] & 16) mask = 15;
    if (!mask) return;
    const bool wide = (reinterpret_cast<uintptr_t>(val) & 15) == 0;   // (the caller's matrix may start at any 8-byte address)
    for (int64_t q = ptr[n] + (t & 7); q < ptr[n + 1]; q += 8)
        for (int k = 0; k < 4; ++k)
            if ((mask >> k) & 1) {
                const bool d = idx[q] == n;
                const double r[4] = {d && k == 0 ? 1.0 : 0.0, d && k == 1 ? 1.0 : 0.0, d && k == 2 ? 1.0 : 0.0, d && k == 3 ? 1.0 : 0.0};
                double* o = val + 16 * q + 4 * k;
                if (wide) {
                    reinterpret_cast<double2*>(o)[0] = make_double2(r[0], r[1]);
                    reinterpret_cast<double2*>(o)[1] = make_double2(r[2], r[3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) o[j] = r[j];
                }
            }
}

void launch_bsr_assembly(const Mesh& m, Args A, double* val, double* Ks, cudaStream_t s) {
    const int64_t next = m.n_nodes() + m.n_hang();
    float* ndv = node_workspace<float>(m, nullptr);
    A.ndv = ndv;
    A.ndt = ndv + 8 * next;
    A.ndf = A.F ? ndv + 16 * next : nullptr;
    if (next > 0) launch_node_prep<float, false>(A, ndv, ndv + 8 * next, (float*)A.ndf, s);
    const int64_t no = (int64_t)m.out_list.size(), nc = (int64_t)m.cut_list.size(), ns = (int64_t)m.sq.size() / 10;
    const int64_t nh = (int64_t)m.sq_hosts.size();
    constexpr int EPB = kOutEpb;
    if (no > 0) jac_out<BSR><<<(unsigned)((no + EPB - 1) / EPB), 8 * EPB, 0, s>>>(A, m.d.out_list, no, nullptr, val, nullptr);
    if (nc > 0)
        jac_cut<BSR><<<(unsigned)nc, 32 * JWPB, 0, s>>>(A, m.d.cut_list, m.d.cut_off, m.d.cut_pts_f, m.d.cut_order, nullptr, val, nullptr);
    if (ns > 0 && nh > 0) {
        cudaMemsetAsync(m.d.slot, 0xff, (size_t)m.n_elem() * sizeof(int32_t), s);
        fill_slots<<<(unsigned)((nh + 255) / 256), 256, 0, s>>>(nh, m.d.sq_hosts, m.d.slot);
        cudaMemsetAsync(Ks, 0, (size_t)nh * 1024 * sizeof(double), s);
        jac_nitsche<FULL><<<(unsigned)((ns + 31) / 32), 32, 0, s>>>(A, m.d.sq_elem, m.d.sq_x, m.d.sq_n, m.d.sq_w, m.d.sq_taub, ns,
                                                                    m.d.slot, Ks, nullptr);
        scatter_kmat<<<(unsigned)((nh * 256 + 255) / 256), 256, 0, s>>>(A, m.d.sq_hosts, nh, Ks, val);
    }
}

}  // namespace

// The Jacobian assembled in 4 x 4 blocks on the mesh's block pattern: val [n_blocks][4][4] float64
// (row component, column component), K = sum_e M_e^T k_e M_e with identity rows for the prescribed
// components; Ks: workspace of 1024 doubles per surface-hosting element.
int bsr_assemble(const Mesh& m, const double* u, const double* up, const double* up2, const double* f,
                 const imga_physics& ph, int precision, const int64_t* bptr, const int32_t* bidx, double* val,
                 double* Ks, void* stream) {
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t nb = (int64_t)m.bsr_idx.size(), nn = m.n_nodes();
    Args A = make_args(m, u, up, up2, f, ph, nullptr, nullptr);
    A.bptr = bptr;
    A.bidx = bidx;
    cudaMemsetAsync(val, 0, (size_t)nb * 16 * sizeof(double), s);
    if (precision == 0) launch_jac64<BSR>(m, A, nullptr, 0, nullptr, val, nullptr, s);
    else launch_bsr_assembly(m, A, val, Ks, s);
    if (nn > 0)
        bsr_strong_rows<<<(unsigned)((8 * nn + 255) / 256), 256, 0, s>>>(nn, bptr, bidx, m.d.bcflag,
                                                                    m.user_bc ? m.d.bcmask_user : nullptr, val);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int element_jacobians(const Mesh& m, const double* u, const double* up, const double* up2, const double* f,
                      const imga_physics& ph, int precision, const int32_t* elems, int64_t n, double* K, void* stream) {
    cudaStream_t s = (cudaStream_t)stream;
    if (n <= 0) return 0;
    Args A = make_args(m, u, up, up2, f, ph, nullptr, nullptr);
    int32_t* slot = m.d.slot;
    cudaMemsetAsync(slot, 0xff, (size_t)m.n_elem() * sizeof(int32_t), s);
    fill_slots<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, elems, slot);
    cudaMemsetAsync(K, 0, (size_t)n * 1024 * sizeof(double), s);
    if (precision == 0) launch_jac64<FULL>(m, A, elems, n, slot, K, nullptr, s);
    else launch_jac<FULL>(m, A, slot, K, nullptr, s);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int block_jacobi_setup(const Mesh& m, const double* u, const double* up, const double* up2, const double* f,
                       const imga_physics& ph, int precision, double* D, double* Dinv, void* stream) {
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t nn = m.n_nodes();
    Args A = make_args(m, u, up, up2, f, ph, nullptr, nullptr);
    cudaMemsetAsync(D, 0, (size_t)nn * 16 * sizeof(double), s);
    if (precision == 0) launch_jac64<DIAG>(m, A, nullptr, 0, nullptr, nullptr, D, s);
    else launch_jac<DIAG>(m, A, nullptr, nullptr, D, s);
    if (nn > 0) {
        jac_strong_rows<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(nn, m.d.bcflag, m.user_bc ? m.d.bcmask_user : nullptr, D);
        bj_invert<<<(unsigned)((nn + 127) / 128), 128, 0, s>>>(nn, D, Dinv);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int block_jacobi_apply(const Mesh& m, const double* Dinv, const double* x, double* y, void* stream) {
    const int64_t nn = m.n_nodes();
    if (nn > 0) bj_apply<<<(unsigned)((nn + 255) / 256), 256, 0, (cudaStream_t)stream>>>(nn, Dinv, x, y);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

}  // namespace imga
