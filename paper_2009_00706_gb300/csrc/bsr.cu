// Matrix-based path: the Jacobian assembled in 4 x 4 blocks (Algorithms 2 and 4: K = sum_e M_e^T
// k_e M_e, identity rows for prescribed components), its product with a vector, and a multilevel
// preconditioner built from it by block coarsening.
//
// Multilevel hierarchy.  Level 0 is the assembled matrix, one block row per node, nodes in Morton
// order.  Level l + 1 aggregates `agg` consecutive block rows of level l (Morton ranges, so aggregates
// stay compact) with a piecewise-constant prolongation P_l per unknown that leaves out the rows of
// level l that are not free (identity rows and empty rows of level 0, dead rows of coarser levels):
//     A_{l+1} = P_l^T A_l P_l,   block (I, J) = sum over i in I, j in J of F_i A_l(i, j) F_j,
// F the diagonal 0/1 mask of free unknowns.  Every row of P has at most one nonzero, so this is a
// block coarsening: no general sparse product.  Since the columns of a fine row are sorted, the fine
// blocks of coarse block (I, J) in fine row i are one contiguous range, and each coarse block is a
// gather in a fixed order (deterministic).  A coarse unknown that no free row reaches (a dead row)
// gets an identity row.  The last level (at most `coarse_max` block rows) is inverted densely.
// One V-cycle applies `nu` damped block-Jacobi sweeps (weight omega), the coarse correction, and `nu`
// sweeps more.  The paper preconditions its Krylov solver with additive Schwarz; its conclusion asks
// for preconditioners suited to the method.  Block coarsening needs only the assembled blocks.
//
// Arithmetic: the hierarchy and the V-cycle run in T = double (plain FP64 path) or T = float (mixed
// path; the assembly itself accumulates in float64).

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "imga_internal.h"

namespace imga {

namespace {

constexpr int kMaxLevels = 24;

// ------------------------------------------------------------------------------------------
// kernels
// ------------------------------------------------------------------------------------------
// Row products of a block matrix, Q quads of lanes per block row.  The blocks come from HBM or L2 (64 or
// 128 bytes each for 32 flops), so what counts is bytes in flight: lane 4 j + i of a row's lanes loads row i
// of block q + j whole (16-byte loads) with the column's vector entry, and kRowAhead steps of Q blocks are
// loaded before the first sum.  Every block's four products are summed by its lane and the blocks' sums
// added in column order by every lane: the order, and the bits, of a thread that walks the row.  Q = 8 (a
// warp per row) shortens the chain where the rows of a level leave the chip idle; from kManyRows on Q = 2,
// which needs a third of the instructions per block.  V-cycle on 74 k nodes, mixed: 349 -> 161 us (137 with
// overlapping launches, see apply(); 5 us more with Q = 1 there, 19 with Q = 4, 9 with twice the steps in flight for Q = 2).
constexpr int kRowAhead = 4;
constexpr int64_t kManyRows = 32768;

// WIDE: 16-byte loads.  The caller's float64 arrays of imga_bsr_spmv may start at any 8-byte address (a view into a
// packed buffer); those that do not start at a 16-byte one are read entry by entry.
template <class T> struct Row4 { T v[4]; };
template <bool WIDE = true, class T> __device__ __forceinline__ Row4<T> load_row(const T* p) {
    Row4<T> r;
    if constexpr (!WIDE) {
#pragma unroll
        for (int k = 0; k < 4; ++k) r.v[k] = __ldg(p + k);
    } else if constexpr (sizeof(T) == 4) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(p));
        r.v[0] = a.x; r.v[1] = a.y; r.v[2] = a.z; r.v[3] = a.w;
    } else {
        const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p) + 1);
        r.v[0] = a.x; r.v[1] = a.y; r.v[2] = b.x; r.v[3] = b.y;
    }
    return r;
}
// (multiply-adds spelled out in one order: the compiler's own choice would depend on the kernel)
template <class T> __device__ __forceinline__ T dot4(const T* a, const T* b) {
    return fma(a[3], b[3], fma(a[2], b[2], fma(a[0], b[0], a[1] * b[1])));
}

// a vector entry of the cycle: x, or x plus the coarse correction of its aggregate on free unknowns
template <class T, bool WIDE = true> struct Plain {
    const T* x;
    __device__ Row4<T> operator()(int64_t c) const {   // (x is rewritten between launches: no read-only loads)
        Row4<T> r;
        if constexpr (!WIDE) {
#pragma unroll
            for (int k = 0; k < 4; ++k) r.v[k] = x[4 * c + k];
        } else if constexpr (sizeof(T) == 4) {
            const float4 a = reinterpret_cast<const float4*>(x)[c];
            r.v[0] = a.x; r.v[1] = a.y; r.v[2] = a.z; r.v[3] = a.w;
        } else {
            const double2 a = reinterpret_cast<const double2*>(x)[2 * c], b = reinterpret_cast<const double2*>(x)[2 * c + 1];
            r.v[0] = a.x; r.v[1] = a.y; r.v[2] = b.x; r.v[3] = b.y;
        }
        return r;
    }
};
template <class T> struct Corrected {
    Plain<T> x, xc;
    const uint8_t* fr;
    uint32_t agg;
    __device__ Row4<T> operator()(int64_t c) const {
        Row4<T> r = x(c);
        const Row4<T> d = xc((uint32_t)c / agg);
        const unsigned f = fr[c];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if ((f >> k) & 1u) r.v[k] += d.v[k];
        return r;
    }
};

// component (lane & 3) of row `row` of A x, on the row's 4 Q lanes (live: this row exists; every lane of the
// warp calls).  begin() runs once, before x is first read: the matrix is loaded ahead of it.
template <int Q, class T, bool WIDE = true, class X, class B>
__device__ __forceinline__ T row_product(bool live, int64_t row, const int64_t* __restrict__ ptr, const int32_t* __restrict__ idx,
                                         const T* __restrict__ val, const X& x, B&& begin) {
    constexpr int D = kRowAhead;   // steps in flight
    const int lane = threadIdx.x & 31, j = (lane >> 2) & (Q - 1), i = lane & 3, first = lane & ~(4 * Q - 1);
    const int64_t q0 = live ? ptr[row] : 0, q1 = live ? ptr[row + 1] : 0;
    T acc = T(0);
    bool begun = false;
    for (int64_t base = q0; __any_sync(0xffffffffu, base < q1); base += Q * D) {
        T t[D];
        int32_t c[D];
        Row4<T> a[D];
#pragma unroll
        for (int g = 0; g < D; ++g) {
            const int64_t q = base + Q * g + j;
            c[g] = -1;
            if (q < q1) {   // (the block does not wait for its column)
                c[g] = __ldg(idx + q);
                a[g] = load_row<WIDE>(val + 16 * q + 4 * i);
            }
        }
        if (!begun) begin();
        begun = true;
#pragma unroll
        for (int g = 0; g < D; ++g) {
            t[g] = T(0);
            if (c[g] >= 0) t[g] = dot4(a[g].v, x(c[g]).v);
        }
#pragma unroll
        for (int g = 0; g < D; ++g)
#pragma unroll
            for (int b = 0; b < Q; ++b) {
                const T s = Q == 1 ? t[g] : __shfl_sync(0xffffffffu, t[g], first + 4 * b + i);
                if (base + Q * g + b < q1) acc += s;
            }
    }
    if (!begun) begin();
    return acc;
}

// y = A x
template <class T, int Q, bool WIDE>
__global__ void __launch_bounds__(256) bsr_mul(int64_t n, const int64_t* __restrict__ ptr, const int32_t* __restrict__ idx,
                                               const T* __restrict__ val, const T* __restrict__ x, T* __restrict__ y) {
    const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / (4 * Q);
    const int l = threadIdx.x & (4 * Q - 1);
    const T acc = row_product<Q, T, WIDE>(row < n, row, ptr, idx, val, Plain<T, WIDE>{x}, [] {});
    if (row < n && l < 4) y[4 * row + l] = acc;
}

// One damped block-Jacobi sweep, out of place: y = x + omega Dinv (b - A x), x with the coarse correction
// where X is Corrected; z (or null): y once more, in float64.
template <class T, class X, int Q>
__global__ void __launch_bounds__(256) ml_sweep(int64_t n, const int64_t* __restrict__ ptr, const int32_t* __restrict__ idx,
                                                const T* __restrict__ val, X x, const T* b,
                                                const T* __restrict__ Dinv, T omega, T* y, double* z) {
    next_may_start();
    const int64_t r0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / (4 * Q);
    const bool live = r0 < n;
    const int64_t row = live ? r0 : n - 1;
    const int l = threadIdx.x & (4 * Q - 1), i = l & 3;
    const Row4<T> D = load_row(Dinv + 16 * row + 4 * i);
    Row4<T> xr;
    T bi;
    const T prod = row_product<Q, T>(live, row, ptr, idx, val, x, [&] {
        after_previous();
        xr = x(row);
        bi = b[4 * row + i];
    });
    const T res = bi - prod;
    T v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __shfl_sync(0xffffffffu, res, (threadIdx.x & 28) | k);
    const T own = i == 0 ? xr.v[0] : i == 1 ? xr.v[1] : i == 2 ? xr.v[2] : xr.v[3];
    const T out = fma(omega, dot4(D.v, v), own);
    if (live && l < 4) {
        y[4 * row + l] = out;
        if (z) z[4 * row + l] = (double)out;
    }
}

// Residual, its restriction and the first sweep of the next level, a block of 256 threads for `per` whole
// aggregates (or one, in turns of 64 / Q rows, if it has more rows): rc[I] = sum of F_i (b - A x)_i over
// the aggregate in row order; xc[I] = omega Dinv_c rc[I] (Dinv_c null: the next level is the dense one,
// which starts from rc alone).  The residual itself is never stored.
template <class T, int Q>
__global__ void __launch_bounds__(256) ml_restrict(int64_t nc, int64_t nf, int agg, int per, const int64_t* __restrict__ ptr,
                                                   const int32_t* __restrict__ idx, const T* __restrict__ val,
                                                   const T* x, const T* b, const uint8_t* __restrict__ fr,
                                                   const T* __restrict__ Dinv_c, T omega, T* rc, T* xc) {
    next_may_start();
    constexpr int R = 64 / Q;   // rows at a time
    __shared__ T s_res[R][4];
    const int r = threadIdx.x / (4 * Q), i = threadIdx.x & 3;
    const int64_t I0 = (int64_t)blockIdx.x * per, I1 = I0 + per < nc ? I0 + per : nc;
    const int64_t i0 = I0 * agg, i1 = I1 * agg < nf ? I1 * agg : nf;
    const int64_t I = I0 + (threadIdx.x >> 2);   // threads 4 a .. 4 a + 3 sum aggregate I0 + a
    T s = T(0);
    for (int64_t a0 = i0; a0 < i1; a0 += R) {
        const int64_t row = a0 + r;
        const bool live = row < i1;
        T bi = T(0);
        const T prod = row_product<Q, T>(live, row, ptr, idx, val, Plain<T>{x}, [&] {
            after_previous();
            if (live) bi = b[4 * row + i];
        });
        const T res = bi - prod;
        if (live && (threadIdx.x & (4 * Q - 1)) < 4) s_res[r][i] = res;
        __syncthreads();
        if (I < I1)
            for (int64_t q = I * agg > a0 ? I * agg : a0; q < (I + 1) * agg && q < a0 + R && q < i1; ++q)
                if ((fr[q] >> i) & 1) s += s_res[q - a0][i];
        __syncthreads();
    }
    after_previous();   // (a block without rows waits too)
    if (I >= I1) return;
    rc[4 * I + i] = s;
    if (!Dinv_c) return;
    T v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __shfl_sync(0xfu << (threadIdx.x & 28), s, (threadIdx.x & 28) | k);
    const Row4<T> D = load_row(Dinv_c + 16 * I + 4 * i);
    xc[4 * I + i] = omega * dot4(D.v, v);
}

// x[i][k] += F_i xc[I(i)][k]: on a level of many rows a pass of its own (the corrected entry at every block,
// with its division by the aggregate size, costs a sweep of 74 k rows 11 us, this pass 3)
template <class T>
__global__ void __launch_bounds__(256) ml_prolong(int64_t nf, uint32_t agg, const uint8_t* __restrict__ fr, const T* xc, T* x) {
    next_may_start();
    after_previous();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i = t >> 2;
    if (i >= nf) return;
    if ((fr[i] >> (t & 3)) & 1) x[t] += xc[4 * ((uint32_t)i / agg) + (t & 3)];
}

// calls f with the quads per row as a constant
template <class F> void with_quads(int64_t rows, F&& f) {
    if (rows >= kManyRows) f(std::integral_constant<int, 2>());
    else f(std::integral_constant<int, 8>());
}

// free mask of level 0 from the assembled float64 matrix: bit k set unless row (node, k) is an
// identity row (diagonal 1, absolute row sum 1) or empty (absolute row sum 0)
__global__ void ml_free0(int64_t n, const int64_t* __restrict__ ptr, const int32_t* __restrict__ idx,
                         const double* __restrict__ val, uint8_t* __restrict__ fr) {
    const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= n) return;
    uint8_t m = 0;
    for (int k = 0; k < 4; ++k) {
        double s = 0.0, d = 0.0;
        for (int64_t q = ptr[row]; q < ptr[row + 1]; ++q) {
            const double* v = val + 16 * q + 4 * k;
            s += fabs(v[0]) + fabs(v[1]) + fabs(v[2]) + fabs(v[3]);
            if (idx[q] == row) d = v[k];
        }
        const bool fixed = (d == 1.0 && s == 1.0) || s == 0.0;
        if (!fixed) m |= (uint8_t)(1 << k);
    }
    fr[row] = m;
}

template <class S, class D>
__global__ void convert_kernel(int64_t n, const S* __restrict__ a, D* __restrict__ b) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = (D)a[i];
}

// coarse block (I, J) = sum over fine rows i of aggregate I and their blocks with column in aggregate J
// of the masked fine block; 16 threads per coarse block, thread (k, m) forms entry (k, m)
template <class T>
__global__ void __launch_bounds__(256) ml_coarsen(int64_t nc, const int64_t* __restrict__ cptr,
                                                  const int32_t* __restrict__ cidx, int64_t nbc, int64_t nf,
                                                  const int64_t* __restrict__ fptr, const int32_t* __restrict__ fidx,
                                                  const T* __restrict__ fval, const uint8_t* __restrict__ ffree, int agg,
                                                  const int64_t* __restrict__ crow, T* __restrict__ cval) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t cb = t >> 4;
    if (cb >= nbc) return;
    const int k = (int)((t >> 2) & 3), mm = (int)(t & 3);
    const int64_t I = crow[cb];
    const int32_t J = cidx[cb];
    const int64_t j0 = (int64_t)J * agg, j1 = j0 + agg;
    double acc = 0.0;
    for (int64_t i = I * agg, iend = (I * agg + agg < nf ? I * agg + agg : nf); i < iend; ++i) {
        if (!((ffree[i] >> k) & 1)) continue;
        int64_t lo = fptr[i], hi = fptr[i + 1];
        while (lo < hi) {   // first column >= j0
            const int64_t mid = (lo + hi) >> 1;
            if (fidx[mid] < j0) lo = mid + 1;
            else hi = mid;
        }
        for (int64_t q = lo; q < fptr[i + 1] && fidx[q] < j1; ++q)
            if ((ffree[fidx[q]] >> mm) & 1) acc += (double)fval[16 * q + 4 * k + mm];
    }
    cval[16 * cb + 4 * k + mm] = (T)acc;
}

// dead rows of a coarse level (no free fine row reaches them) get an identity row; fr = the rest
template <class T>
__global__ void ml_dead(int64_t n, const int64_t* __restrict__ ptr, const int64_t* __restrict__ diag,
                        T* __restrict__ val, uint8_t* __restrict__ fr) {
    const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= n) return;
    uint8_t m = 0;
    for (int k = 0; k < 4; ++k) {
        T s = T(0);
        for (int64_t q = ptr[row]; q < ptr[row + 1]; ++q) {
            const T* v = val + 16 * q + 4 * k;
            s += fabs(v[0]) + fabs(v[1]) + fabs(v[2]) + fabs(v[3]);
        }
        if (s == T(0)) val[16 * diag[row] + 5 * k] = T(1);
        else m |= (uint8_t)(1 << k);
    }
    fr[row] = m;
}

// inverse of every diagonal block (Gauss-Jordan with partial pivoting in float64); a block whose
// pivot falls below 1e-14 of its largest entry is replaced by the identity
template <class T>
__global__ void ml_diag_inv(int64_t n, const int64_t* __restrict__ diag, const T* __restrict__ val, T* __restrict__ Dinv) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    double a[4][8];
    double scale = 0.0;
    const T* v = val + 16 * diag[r];
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) {
            a[i][j] = (double)v[4 * i + j];
            a[i][4 + j] = i == j ? 1.0 : 0.0;
            scale = fmax(scale, fabs(a[i][j]));
        }
    bool ok = scale > 0.0;
    for (int col = 0; col < 4 && ok; ++col) {
        int piv = col;
        for (int i = col + 1; i < 4; ++i)
            if (fabs(a[i][col]) > fabs(a[piv][col])) piv = i;
        if (!(fabs(a[piv][col]) > 1e-14 * scale)) { ok = false; break; }
        if (piv != col)
            for (int j = 0; j < 8; ++j) { const double t = a[col][j]; a[col][j] = a[piv][j]; a[piv][j] = t; }
        const double inv = 1.0 / a[col][col];
        for (int j = 0; j < 8; ++j) a[col][j] *= inv;
        for (int i = 0; i < 4; ++i) {
            if (i == col) continue;
            const double f = a[i][col];
            if (f != 0.0)
                for (int j = 0; j < 8; ++j) a[i][j] -= f * a[col][j];
        }
    }
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) Dinv[16 * r + 4 * i + j] = (T)(ok ? a[i][4 + j] : (i == j ? 1.0 : 0.0));
}

// dense copy [N][N] (N = 4 n) of the last level; an all-zero row gets a 1 on the diagonal
template <class T>
__global__ void ml_densify(int64_t n, const int64_t* __restrict__ ptr, const int32_t* __restrict__ idx,
                           const T* __restrict__ val, double* __restrict__ dense) {
    const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= n) return;
    const int64_t N = 4 * n;
    for (int k = 0; k < 4; ++k) {
        double* d = dense + (4 * row + k) * N;
        for (int64_t j = 0; j < N; ++j) d[j] = 0.0;
        double s = 0.0;
        for (int64_t q = ptr[row]; q < ptr[row + 1]; ++q)
            for (int mm = 0; mm < 4; ++mm) {
                const double x = (double)val[16 * q + 4 * k + mm];
                d[4 * (int64_t)idx[q] + mm] = x;
                s += fabs(x);
            }
        if (s == 0.0) d[4 * row + k] = 1.0;
    }
}

// Inverse of the dense N x N matrix by Gauss-Jordan with partial pivoting, one block, the
// augmented [A | I] in shared memory (float64).  A singular column leaves *bad set and the identity.
template <class T>
__global__ void __launch_bounds__(512) ml_dense_inverse(int N, const double* __restrict__ A, T* __restrict__ Ainv,
                                                        int* __restrict__ bad) {
    extern __shared__ double sa[];   // [N][2N]
    __shared__ int s_piv;
    __shared__ double s_scale;
    const int W = 2 * N;
    for (int t = threadIdx.x; t < N * W; t += blockDim.x) {
        const int i = t / W, j = t % W;
        sa[t] = j < N ? A[(int64_t)i * N + j] : (j - N == i ? 1.0 : 0.0);
    }
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int t = 0; t < N * N; ++t) s = fmax(s, fabs(A[t]));
        s_scale = s;
    }
    __syncthreads();
    bool ok = true;
    for (int col = 0; col < N; ++col) {
        if (threadIdx.x == 0) {
            int p = col;
            for (int i = col + 1; i < N; ++i)
                if (fabs(sa[i * W + col]) > fabs(sa[p * W + col])) p = i;
            s_piv = fabs(sa[p * W + col]) > 1e-300 + 1e-15 * s_scale ? p : -1;
        }
        __syncthreads();
        const int p = s_piv;
        if (p < 0) { ok = false; break; }
        if (p != col)
            for (int j = threadIdx.x; j < W; j += blockDim.x) {
                const double t = sa[col * W + j];
                sa[col * W + j] = sa[p * W + j];
                sa[p * W + j] = t;
            }
        __syncthreads();
        const double inv = 1.0 / sa[col * W + col];
        __syncthreads();
        for (int j = threadIdx.x; j < W; j += blockDim.x) sa[col * W + j] *= inv;
        __syncthreads();
        for (int t = threadIdx.x; t < N * W; t += blockDim.x) {
            const int i = t / W, j = t % W;
            if (i == col || j == col) continue;
            const double f = sa[i * W + col];
            if (f != 0.0) sa[t] -= f * sa[col * W + j];
        }
        __syncthreads();
        for (int i = threadIdx.x; i < N; i += blockDim.x)
            if (i != col) sa[i * W + col] = 0.0;
        __syncthreads();
    }
    if (!ok && threadIdx.x == 0) *bad = 1;
    for (int t = threadIdx.x; t < N * N; t += blockDim.x) {
        const int i = t / N, j = t % N;
        Ainv[t] = (T)(ok ? sa[i * W + N + j] : (i == j ? 1.0 : 0.0));
    }
}

// r in the cycle's precision and the first sweep from x = 0: x = omega Dinv r
template <class T>
__global__ void ml_start(int64_t n, const T* __restrict__ Dinv, T omega, const double* rd, T* r, T* x) {
    next_may_start();
    after_previous();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t row = t >> 2;
    const int i = (int)(t & 3);
    if (row >= n) return;
    const T own = (T)rd[t];
    T v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __shfl_sync(0xfu << (threadIdx.x & 28), own, (threadIdx.x & 28) | k);
    r[t] = own;
    const Row4<T> D = load_row(Dinv + 16 * row + 4 * i);
    x[t] = omega * dot4(D.v, v);
}

// y = Ainv r for the dense last level (N <= 4 * coarse_max <= 96), one block, a thread per row: r from
// shared memory, 8 entries of the row loaded before they are added (one serial load per entry was its time)
template <class T>
__global__ void __launch_bounds__(96) ml_dense_apply(int N, const T* __restrict__ Ainv, const T* r, T* y) {
    next_may_start();
    after_previous();
    __shared__ T s_r[96];
    const int i = threadIdx.x;
    if (i < N) s_r[i] = r[i];
    __syncthreads();
    if (i >= N) return;
    T s = T(0);
    const T* a = Ainv + (int64_t)i * N;
#pragma unroll 8
    for (int j = 0; j < N; ++j) s += a[j] * s_r[j];
    y[i] = s;
}

inline unsigned blocks(int64_t threads, int per = 256) { return (unsigned)std::max<int64_t>(1, (threads + per - 1) / per); }

}  // namespace

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
struct MLPattern {
    int64_t n = 0;                  // block rows
    std::vector<int64_t> ptr;       // [n + 1]
    std::vector<int32_t> idx;
    int64_t *dptr = nullptr, *ddiag = nullptr, *drow = nullptr;   // device: pattern, diagonal position, row of each block
    int32_t* didx = nullptr;
};

template <class T>
struct MLValues {
    T* A[kMaxLevels] = {};
    T* Dinv[kMaxLevels] = {};
    T *r[kMaxLevels] = {}, *x[kMaxLevels] = {}, *res[kMaxLevels] = {};
    T* Cinv = nullptr;
    bool alloc = false;
};

struct Multilevel {
    int agg = 0, coarse_max = 0;
    std::vector<MLPattern> lev;     // lev.back() is the dense level
    uint8_t* fr[kMaxLevels] = {};   // free masks per level (device)
    double* A0 = nullptr;           // assembled fine matrix, float64
    double* Ks = nullptr;           // surface element matrices (assembly workspace)
    double* dense = nullptr;        // [N][N] last level, float64
    int* bad = nullptr;
    MLValues<double> vd;
    MLValues<float> vf;
    int precision = -1;             // precision of the last setup
    int nu = 1;
    double omega = 0.5;
};

namespace {

template <class T>
void free_values(MLValues<T>& v, size_t nlev) {
    for (size_t l = 0; l < nlev; ++l) {
        if (l > 0 || !std::is_same<T, double>::value) cudaFree(v.A[l]);
        cudaFree(v.Dinv[l]); cudaFree(v.r[l]); cudaFree(v.x[l]); cudaFree(v.res[l]);
    }
    cudaFree(v.Cinv);
    v = MLValues<T>();
}

// the coarse pattern of aggregating `agg` consecutive block rows and columns
void coarsen_pattern(const MLPattern& f, int agg, MLPattern& c) {
    c.n = (f.n + agg - 1) / agg;
    c.ptr.assign(c.n + 1, 0);
    std::vector<std::vector<int32_t>> rows(c.n);
#pragma omp parallel for schedule(dynamic, 256)
    for (int64_t I = 0; I < c.n; ++I) {
        std::vector<int32_t>& cols = rows[I];
        for (int64_t i = I * agg; i < std::min<int64_t>(I * agg + agg, f.n); ++i)
            for (int64_t q = f.ptr[i]; q < f.ptr[i + 1]; ++q) cols.push_back(f.idx[q] / agg);
        std::sort(cols.begin(), cols.end());
        cols.erase(std::unique(cols.begin(), cols.end()), cols.end());
    }
    for (int64_t I = 0; I < c.n; ++I) c.ptr[I + 1] = c.ptr[I] + (int64_t)rows[I].size();
    c.idx.resize(c.ptr[c.n]);
#pragma omp parallel for schedule(dynamic, 256)
    for (int64_t I = 0; I < c.n; ++I) std::copy(rows[I].begin(), rows[I].end(), c.idx.begin() + c.ptr[I]);
}

bool upload_pattern(MLPattern& p, std::string& err) {
    const int64_t nb = p.ptr.back();
    std::vector<int64_t> diag(std::max<int64_t>(1, p.n), -1), row(std::max<int64_t>(1, nb), 0);
    for (int64_t i = 0; i < p.n; ++i)
        for (int64_t q = p.ptr[i]; q < p.ptr[i + 1]; ++q) {
            row[q] = i;
            if (p.idx[q] == i) diag[i] = q;
        }
    for (int64_t i = 0; i < p.n; ++i)
        if (diag[i] < 0) { err = "block pattern without a diagonal block"; return false; }
    auto up = [&](auto** d, const auto& v) {
        using E = typename std::remove_reference<decltype(v)>::type::value_type;
        const size_t bytes = std::max<size_t>(1, v.size()) * sizeof(E);
        if (cudaMalloc((void**)d, bytes) != cudaSuccess) return false;
        return v.empty() || cudaMemcpy(*d, v.data(), v.size() * sizeof(E), cudaMemcpyHostToDevice) == cudaSuccess;
    };
    if (!up(&p.dptr, p.ptr) || !up(&p.didx, p.idx) || !up(&p.ddiag, diag) || !up(&p.drow, row)) {
        err = "multilevel pattern upload failed";
        cudaGetLastError();
        return false;
    }
    return true;
}

template <class T>
MLValues<T>& values(Multilevel& L);
template <> MLValues<double>& values<double>(Multilevel& L) { return L.vd; }
template <> MLValues<float>& values<float>(Multilevel& L) { return L.vf; }

template <class T>
bool alloc_values(Multilevel& L, std::string& err) {
    MLValues<T>& v = values<T>(L);
    if (v.alloc) return true;
    const size_t nl = L.lev.size();
    bool ok = true;
    for (size_t l = 0; l < nl && ok; ++l) {
        const MLPattern& p = L.lev[l];
        const int64_t nb = p.ptr.back(), n = std::max<int64_t>(1, p.n);
        if (l == 0 && std::is_same<T, double>::value) v.A[0] = (T*)L.A0;
        else ok = ok && cudaMalloc((void**)&v.A[l], std::max<int64_t>(1, nb) * 16 * sizeof(T)) == cudaSuccess;
        ok = ok && cudaMalloc((void**)&v.Dinv[l], n * 16 * sizeof(T)) == cudaSuccess &&
             cudaMalloc((void**)&v.r[l], n * 4 * sizeof(T)) == cudaSuccess &&
             cudaMalloc((void**)&v.x[l], n * 4 * sizeof(T)) == cudaSuccess &&
             cudaMalloc((void**)&v.res[l], n * 4 * sizeof(T)) == cudaSuccess;
    }
    const int64_t N = 4 * L.lev.back().n;
    ok = ok && cudaMalloc((void**)&v.Cinv, std::max<int64_t>(1, N * N) * sizeof(T)) == cudaSuccess;
    if (!ok) { err = "multilevel allocation failed"; cudaGetLastError(); return false; }
    v.alloc = true;
    return true;
}

template <class T>
int setup_values(const Mesh& m, Multilevel& L, cudaStream_t s) {
    MLValues<T>& v = values<T>(L);
    const size_t nl = L.lev.size();
    const MLPattern& p0 = L.lev[0];
    if (!std::is_same<T, double>::value)
        convert_kernel<double, T><<<blocks(16 * p0.ptr.back()), 256, 0, s>>>(16 * p0.ptr.back(), L.A0, v.A[0]);
    for (size_t l = 0; l + 1 < nl; ++l) {
        const MLPattern &f = L.lev[l], &c = L.lev[l + 1];
        ml_diag_inv<T><<<blocks(f.n, 128), 128, 0, s>>>(f.n, f.ddiag, v.A[l], v.Dinv[l]);
        const int64_t nbc = c.ptr.back();
        ml_coarsen<T><<<blocks(16 * nbc), 256, 0, s>>>(c.n, c.dptr, c.didx, nbc, f.n, f.dptr, f.didx, v.A[l], L.fr[l],
                                                         L.agg, c.drow, v.A[l + 1]);
        ml_dead<T><<<blocks(c.n), 256, 0, s>>>(c.n, c.dptr, c.ddiag, v.A[l + 1], L.fr[l + 1]);
    }
    const MLPattern& d = L.lev.back();
    const int N = (int)(4 * d.n);
    if (N > 0) {
        ml_densify<T><<<blocks(d.n), 256, 0, s>>>(d.n, d.dptr, d.didx, v.A[nl - 1], L.dense);
        const size_t smem = (size_t)N * 2 * N * sizeof(double);
        ml_dense_inverse<T><<<1, 512, smem, s>>>(N, L.dense, v.Cinv, L.bad);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

// V-cycle below the first sweep of level l (x[l] = omega Dinv r[l] is there); the result is in *out, one of
// the level's two iterates.  z (level 0, or null): the last sweep also writes it there in float64.
template <class T>
void vcycle(Multilevel& L, size_t l, Chain& go, T** out, double* z) {
    MLValues<T>& v = values<T>(L);
    const MLPattern& p = L.lev[l];
    const T om = (T)L.omega;
    T *x = v.x[l], *y = v.res[l];
    auto sweep = [&](auto in, double* zk) {
        with_quads(p.n, [&](auto q) {
            constexpr int Q = decltype(q)::value;
            go(ml_sweep<T, decltype(in), Q>, blocks(4 * Q * p.n), 256, 0, p.n, p.dptr, p.didx, v.A[l], in, v.r[l], v.Dinv[l], om, y, zk);
        });
        std::swap(x, y);
    };
    for (int k = 1; k < L.nu; ++k) sweep(Plain<T>{x}, nullptr);
    const MLPattern& c = L.lev[l + 1];
    const bool dense = l + 2 == L.lev.size();
    with_quads(p.n, [&](auto q) {
        constexpr int Q = decltype(q)::value;
        const int per = std::max(1, 64 / Q / L.agg);
        go(ml_restrict<T, Q>, (c.n + per - 1) / per, 256, 0, c.n, p.n, L.agg, per, p.dptr, p.didx, v.A[l], x, v.r[l], L.fr[l],
           dense ? nullptr : v.Dinv[l + 1], om, v.r[l + 1], v.x[l + 1]);
    });
    T* xc = v.x[l + 1];
    if (dense) go(ml_dense_apply<T>, 1, 96, 0, (int)(4 * c.n), v.Cinv, v.r[l + 1], xc);
    else vcycle<T>(L, l + 1, go, &xc, nullptr);
    for (int k = 0; k < L.nu; ++k) {
        double* zk = k + 1 == L.nu ? z : nullptr;
        if (k == 0 && p.n < kManyRows) {
            sweep(Corrected<T>{{x}, {xc}, L.fr[l], (uint32_t)L.agg}, zk);
            continue;
        }
        if (k == 0) go(ml_prolong<T>, blocks(4 * p.n), 256, 0, p.n, (uint32_t)L.agg, L.fr[l], xc, x);
        sweep(Plain<T>{x}, zk);
    }
    *out = x;
}

// z = V-cycle(r): two launches per level (three where it has many rows) and one for the dense one (six before).
// On the small levels a launch is little more than its own latency (4 us for 12 k rows): with Chain the next
// one's blocks are there early and have their part of the matrix loaded when this one ends.  12 launches on 74 k
// nodes: 161 -> 137 us.
template <class T>
void apply(Multilevel& L, const double* r, double* z, cudaStream_t s) {
    MLValues<T>& v = values<T>(L);
    const int64_t n = L.lev[0].n;
    if (L.lev.size() == 1) {   // dense only
        convert_kernel<double, T><<<blocks(4 * n), 256, 0, s>>>(4 * n, r, v.r[0]);
        ml_dense_apply<T><<<1, 96, 0, s>>>((int)(4 * n), v.Cinv, v.r[0], v.x[0]);
        convert_kernel<T, double><<<blocks(4 * n), 256, 0, s>>>(4 * n, v.x[0], z);
        return;
    }
    Chain go(s);
    go(ml_start<T>, blocks(4 * n), 256, 0, n, v.Dinv[0], (T)L.omega, r, v.r[0], v.x[0]);
    T* x;
    vcycle<T>(L, 0, go, &x, z);
}

}  // namespace

void multilevel_free(Mesh& m) {
    Multilevel* L = (Multilevel*)m.mlev;
    if (!L) return;
    free_values(L->vd, L->lev.size());
    free_values(L->vf, L->lev.size());
    for (auto& p : L->lev) { cudaFree(p.dptr); cudaFree(p.didx); cudaFree(p.ddiag); cudaFree(p.drow); }
    for (int l = 0; l < kMaxLevels; ++l) cudaFree(L->fr[l]);
    cudaFree(L->A0); cudaFree(L->Ks); cudaFree(L->dense); cudaFree(L->bad);
    delete L;
    m.mlev = nullptr;
}

// Patterns of the hierarchy (host, once per mesh and (agg, coarse_max)) and the device arrays.
int multilevel_prepare(Mesh& m, int agg, int coarse_max, std::string& err) {
    Multilevel* L = (Multilevel*)m.mlev;
    if (L && L->agg == agg && L->coarse_max == coarse_max) return 0;
    multilevel_free(m);
    if (agg < 2 || coarse_max < 1 || 4 * coarse_max > 96) { err = "multilevel: agg >= 2 and 1 <= coarse_max <= 24"; return 1; }
    if (m.bsr_ptr.empty()) build_bsr_pattern(m);
    L = new Multilevel();
    m.mlev = L;
    L->agg = agg;
    L->coarse_max = coarse_max;
    MLPattern p0;
    p0.n = m.n_nodes();
    p0.ptr = m.bsr_ptr;
    p0.idx = m.bsr_idx;
    L->lev.push_back(std::move(p0));
    while (L->lev.back().n > coarse_max) {
        if ((int)L->lev.size() >= kMaxLevels) { err = "multilevel: too many levels"; multilevel_free(m); return 1; }
        MLPattern c;
        coarsen_pattern(L->lev.back(), agg, c);
        L->lev.push_back(std::move(c));
    }
    for (auto& p : L->lev)
        if (!upload_pattern(p, err)) { multilevel_free(m); return 1; }
    const int64_t N = 4 * L->lev.back().n;
    bool ok = cudaMalloc((void**)&L->A0, std::max<int64_t>(1, m.bsr_ptr.back()) * 16 * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&L->Ks, std::max<size_t>(1, m.sq_hosts.size()) * 1024 * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&L->dense, std::max<int64_t>(1, N * N) * sizeof(double)) == cudaSuccess &&
              cudaMalloc((void**)&L->bad, sizeof(int)) == cudaSuccess;
    for (size_t l = 0; l < L->lev.size() && ok; ++l)
        ok = cudaMalloc((void**)&L->fr[l], std::max<int64_t>(1, L->lev[l].n)) == cudaSuccess;
    if (!ok) { err = "multilevel allocation failed"; cudaGetLastError(); multilevel_free(m); return 1; }
    cudaMemset(L->bad, 0, sizeof(int));
    // the dense inverse keeps [N][2N] doubles in shared memory
    const int smem = (int)(N * 2 * N * sizeof(double));
    cudaFuncSetAttribute(ml_dense_inverse<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, std::max(smem, 1));
    cudaFuncSetAttribute(ml_dense_inverse<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, std::max(smem, 1));
    return 0;
}

// Assemble the fine matrix at the state (u, ...) and build every level's values in the precision.
int multilevel_setup(Mesh& m, const double* u, const double* up, const double* up2, const double* f,
                     const imga_physics& ph, int precision, int nu, double omega, void* stream, std::string& err) {
    Multilevel* L = (Multilevel*)m.mlev;
    if (!L) { err = "multilevel: not prepared"; return 1; }
    cudaStream_t s = (cudaStream_t)stream;
    L->nu = std::max(1, nu);
    L->omega = omega;
    L->precision = precision;
    const MLPattern& p0 = L->lev[0];
    if (bsr_assemble(m, u, up, up2, f, ph, precision, p0.dptr, p0.didx, L->A0, L->Ks, s)) { err = "assembly failed"; return 1; }
    ml_free0<<<blocks(p0.n), 256, 0, s>>>(p0.n, p0.dptr, p0.didx, L->A0, L->fr[0]);
    if (precision == 0) {
        if (!alloc_values<double>(*L, err)) return 1;
        return setup_values<double>(m, *L, s) ? (err = "multilevel setup launch failed", 1) : 0;
    }
    if (!alloc_values<float>(*L, err)) return 1;
    return setup_values<float>(m, *L, s) ? (err = "multilevel setup launch failed", 1) : 0;
}

// z = V-cycle(r), float64 vectors [n_nodes][4]
int multilevel_apply(Mesh& m, const double* r, double* z, void* stream) {
    Multilevel* L = (Multilevel*)m.mlev;
    if (!L || L->precision < 0) return 1;
    cudaStream_t s = (cudaStream_t)stream;
    if (L->lev[0].n == 0) return 0;
    if (L->precision == 0) apply<double>(*L, r, z, s);
    else apply<float>(*L, r, z, s);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

// block rows per level (host array of n_levels entries, may be null) and whether the dense
// inverse met a singular pivot; returns the number of levels
int multilevel_info(Mesh& m, int64_t* rows, int* singular) {
    Multilevel* L = (Multilevel*)m.mlev;
    if (!L) return 0;
    if (rows)
        for (size_t l = 0; l < L->lev.size(); ++l) rows[l] = L->lev[l].n;
    if (singular) {
        int h = 0;
        cudaMemcpy(&h, L->bad, sizeof(int), cudaMemcpyDeviceToHost);
        *singular = h;
    }
    return (int)L->lev.size();
}

// y = A x with the assembled float64 matrix val on the mesh's block pattern
int bsr_spmv(Mesh& m, const double* val, const double* x, double* y, void* stream, std::string& err) {
    if (m.bsr_ptr.empty()) build_bsr_pattern(m);
    Multilevel* L = (Multilevel*)m.mlev;
    if (!L) { err = "the block pattern is not on the device (call the assembly first)"; return 1; }
    const MLPattern& p = L->lev[0];
    const bool wide = (((uintptr_t)val | (uintptr_t)x) & 15) == 0;
    if (p.n > 0)
        with_quads(p.n, [&](auto q) {
            constexpr int Q = decltype(q)::value;
            auto run = [&](auto kernel) { kernel<<<blocks(4 * Q * p.n), 256, 0, (cudaStream_t)stream>>>(p.n, p.dptr, p.didx, val, x, y); };
            if (wide) run(bsr_mul<double, Q, true>);
            else run(bsr_mul<double, Q, false>);
        });
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

// the assembled float64 fine matrix of the hierarchy (valid after multilevel_setup)
double* multilevel_matrix(Mesh& m) { return m.mlev ? ((Multilevel*)m.mlev)->A0 : nullptr; }

// the device pattern of level 0 (prepared on first use with default hierarchy parameters)
int bsr_device_pattern(Mesh& m, const int64_t** ptr, const int32_t** idx, double** ks, std::string& err) {
    if (!m.mlev && multilevel_prepare(m, 6, 16, err)) return 1;
    Multilevel* L = (Multilevel*)m.mlev;
    *ptr = L->lev[0].dptr;
    *idx = L->lev[0].didx;
    *ks = L->Ks;
    return 0;
}

}  // namespace imga
