// VMS residual R(u) and Jacobian-vector product J(u) v on Q1 octree elements.
//
// Weak form: Eqs. (ALE-VMS-form) and (vms), fine scales Eqs. (uprime) and (pprime), Nitsche
// terms Eq. (weakbc); In elements skipped, Out elements on the 2x2x2 Gauss rule, Intercepted
// elements on their adaptive sub-cell points (Algorithm 1); element vectors scattered to the
// nodes through the hanging-node operator M_e^T (Algorithms 2 and 3).
//
// Every quadrature point is reduced to 16 coefficients: with w = phi_a e_i and q = phi_a,
//     r_{a,i} += wq [ phi_a F_i + d_j phi_a S_ij ],     r_{a,p} += wq [ phi_a G + d_j phi_a H_j ],
//   F_i  = rho (du_i/dt + (u.grad u)_i - f_i) + (u'.grad u)_i                    terms 1, 6, -F
//   S_ij = sigma_ij - u'_i u_j - p' delta_ij - u'_i u'_j / rho + taubar (u'.grad u)_i u'_j
//                                                                                terms 2, 4, 5, 7, 8
//   G    = div u,   H_j = -u'_j / rho                                             terms 3, 4
// J v is the forward-mode derivative of the same code (dual numbers value + tangent): the
// matrix of Algorithms 2/4 applied to v without being formed.
//
// Kernels (T = float or double element arithmetic, nodal gathers always float64, scatter into slots
// that node_gather sums, or by float64 atomics):
//   vms_interior  8 threads per Out element: thread c gathers corner c, evaluates Gauss point c,
//                 then contracts node c's four rows over the 8 points; interpolation and test
//                 functions both run in the monomial form of the trilinear basis.
//                 float64: interior_element64, the same with fewer FP64 instructions.
//   vms_cut       one warp per Intercepted element; lane l evaluates sub-cell points l, l + 32, ...
//                 and accumulates their monomial moments, summed over the lanes at the end;
//   vms_cut_split four warps per element where elements are few, vms_cut64 in float64.
//   nitsche       one thread per surface point, for elements hosting few points;
//   nitsche_el    one warp per element hosting many, lanes over its points (moments).
//   strong_rows   Dirichlet rows U - g and In-only rows, written after every scatter.

#include <cuda_runtime.h>

#include <cstdio>
#include <algorithm>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>

#include "imga_internal.h"
#include "vms_device.cuh"

namespace imga {

namespace {

// ------------------------------------------------------------------------------------------
// Out elements: 8 threads per element
// ------------------------------------------------------------------------------------------
template <class T> struct Epb { static constexpr int value = 16; };   // elements per block

template <class T> struct IntShape {
    static constexpr int EPB = Epb<T>::value;                                   // elements per block
    static constexpr int THREADS = 8 * EPB;
    // element stride of the corner rows: 8 rows of CS plus 8 T, so the elements of a warp start 8
    // (float) or 16 (double) banks apart and column and broadcast row reads are conflict-free
    static constexpr int ESTR = 8 * CS + 8;
    static constexpr int MSTR = 32 + 16 / (int)sizeof(T);   // row stride of the per-point moments
    static constexpr size_t smem = (size_t)(2 * EPB * ESTR + EPB * 8 * MSTR) * sizeof(T);
};

// generic / GEN: the float64 evaluations of a mixed-precision solve (its residuals and the J v of its restarts) run
// their volume kernels on the generic element code instead of the ones below.  Such a solve turns the last bit of a
// residual into float32 steps of its preconditioner and matvecs, and those into differences as large as its
// tolerance (1e-9 to 1e-7 of u at 1e-8): with other roundings it would end at another solution, no nearer and no
// further from the root.  So this keeps the solutions that a given mesh and state have had; it is no matter of
// accuracy, and such a residual differs in its last bits from the one imga_residual returns.  It costs a solve of the
// 7.3 k element sphere 1.5 of 35 ms; at 2.0 M elements a float64 J v of the Out elements takes 20.7 ms this way, 11.2 by
// interior_element64.  (The penalty with a velocity per surface point has one kernel for all callers.)
//
// One Out element in float64 on 8 lanes of a warp (c = lane & 7); nd its 8 corner rows, sw the warp's
// 4 x 272 doubles.  FP64 instructions are the cost (see Const64), so the work goes to lanes by what
// shares most of them:
//   1. a lane takes one column (u, v, w, p and, J v, their tangents; R: the du/dt columns) of all 8
//      corners: Hadamard transform, then the inverse along z, y, x with the Gauss abscissa in its
//      multiply-adds, whose intermediates are the gradients and mixed derivatives (62 instructions for
//      8 points; point by point they are 8 + 12 + 4 per point).  du/dt of J v: shuffles (6 per column).
//   2. a lane takes Gauss point c: pointwise64.
//   3. a lane takes component c & 3 and the four points of one z side: the transposed sums along x and
//      y, then z with its partner lane (52 instructions).
// 283 k elements (sphere wake), one R and one J v with all their kernels: 5.91 -> 3.88 ms.
template <bool JV>
__device__ __forceinline__ void interior_element64(const Args& A, const double* nd, double* sw, int lane, int64_t idx,
                                                   bool valid, int lv, int prob, int32_t id) {
    constexpr double gam = kGauss;
    const int c = lane & 7;
    double* E = sw + (lane >> 3) * 272;   // V [8 columns][8], GX | GY | GZ [8][4], XY | XZ | YZ [8][2]
    __syncwarp();
    {
        const int col = JV ? (c & 3) + (c >> 2) * CT : (c < 7 ? c : 6);
        double a[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) a[t] = nd[t * CS + col];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if (!(t & (1 << k))) {
                    const double lo = a[t], hi = a[t | (1 << k)];
                    a[t] = lo + hi;
                    a[t | (1 << k)] = hi - lo;
                }
        double *V = E + 8 * c, *GX = E + 64 + 4 * c, *GY = E + 96 + 4 * c, *GZ = E + 128 + 4 * c, *XY = E + 160 + 2 * c,
               *XZ = E + 176 + 2 * c, *YZ = E + 192 + 2 * c;
#pragma unroll
        for (int z = 0; z < 2; ++z) {
            const double gz = z ? gam : -gam;
            double b[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) b[t] = fma(gz, a[4 + t], a[t]);
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                const double gy = y ? gam : -gam;
                const double c0 = fma(gy, b[2], b[0]), c1 = fma(gy, b[3], b[1]);
                V[4 * z + 2 * y] = fma(-gam, c1, c0);
                V[4 * z + 2 * y + 1] = fma(gam, c1, c0);
                GX[2 * z + y] = c1;
            }
            GY[2 * z] = fma(-gam, b[3], b[2]);
            GY[2 * z + 1] = fma(gam, b[3], b[2]);
            XY[z] = b[3];
        }
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const double gy = y ? gam : -gam;
            const double d0 = fma(gy, a[6], a[4]), d1 = fma(gy, a[7], a[5]);
            GZ[2 * y] = fma(-gam, d1, d0);
            GZ[2 * y + 1] = fma(gam, d1, d0);
            XZ[y] = d1;
        }
        YZ[0] = fma(-gam, a[7], a[6]);
        YZ[1] = fma(gam, a[7], a[6]);
    }
    // 8 x the value at Gauss point c of a field whose value at corner c this lane holds
    auto to_point = [&](double x) {
#pragma unroll
        for (int k = 0; k < 3; ++k) x = fma(1.0 + gam, x, (1.0 - gam) * __shfl_xor_sync(0xffffffffu, x, 1 << k));
        return x;
    };
    Point64 F;
    if (JV)
        for (int i = 0; i < 3; ++i) F.a[i] = to_point(nd[c * CS + 4 + i]);
    if (A.ndf)
        for (int i = 0; i < 3; ++i) F.f[i] = to_point(nd[c * CS + CF + i]);
    __syncwarp();
    const int x = c & 1, y = (c >> 1) & 1, z = c >> 2, yz = c >> 1, xz = x | (z << 1), xy = c & 3;
    Tangent64 D;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const double v = E[8 * i + c], gx = E[64 + 4 * i + yz], gy = E[96 + 4 * i + xz], gz = E[128 + 4 * i + xy];
        if (i < 3) { F.u[i] = v; F.G[i][0] = gx; F.G[i][1] = gy; F.G[i][2] = gz; }
        else { F.p = v; F.gp[0] = gx; F.gp[1] = gy; F.gp[2] = gz; }
    }
    if (!JV)
        for (int i = 0; i < 3; ++i) F.a[i] = E[8 * (4 + i) + c];
    auto mixed = [&](int b, double H[3]) {   // (grad div u)_i = sum_{j != i} d_i d_j u_j
        H[0] = E[160 + 2 * (b + 1) + z] + E[176 + 2 * (b + 2) + y];
        H[1] = E[160 + 2 * b + z] + E[192 + 2 * (b + 2) + x];
        H[2] = E[176 + 2 * b + y] + E[192 + 2 * (b + 1) + x];
    };
    mixed(0, F.H);
    if (JV) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double v = E[8 * (4 + i) + c], gx = E[64 + 4 * (4 + i) + yz], gy = E[96 + 4 * (4 + i) + xz],
                         gz = E[128 + 4 * (4 + i) + xy];
            if (i < 3) { D.u[i] = v; D.G[i][0] = gx; D.G[i][1] = gy; D.G[i][2] = gz; }
            else { D.p = v; D.gp[0] = gx; D.gp[1] = gy; D.gp[2] = gz; }
        }
        mixed(4, D.H);
    }
    double W[16];
    {
        const Phys<double> P(A, prob);
        const Const64 C(A, P, lv, A.lc[lv][4], A.lc[lv][5]);
        pointwise64<JV>(C, A.ndf != nullptr, A.c0th, F, D, W);
    }
    __syncwarp();   // every lane has read its fields: the coefficients [16][8] take their place
#pragma unroll
    for (int k = 0; k < 16; ++k) E[8 * k + c] = W[k];
    __syncwarp();
    // the four points of side z = hz: sums along x, then y, for every S over (x, y): M, and Z the sums of
    // the z coefficient
    const int k = c & 3, hz = c >> 2;
    double M[4], Z[4];
    {
        const double *f = E + 8 * k + 4 * hz, *sx = E + 8 * (4 + 3 * k) + 4 * hz, *sy = sx + 8, *sz = sx + 16;
        double lo[2], hi[2], ylo[2], yhi[2], zlo[2], zhi[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const double f0 = f[2 * q], f1 = f[2 * q + 1];
            lo[q] = f0 + f1;
            hi[q] = (f1 + sx[2 * q + 1]) + (sx[2 * q] - f0);
            ylo[q] = sy[2 * q] + sy[2 * q + 1];
            yhi[q] = sy[2 * q + 1] - sy[2 * q];
            zlo[q] = sz[2 * q] + sz[2 * q + 1];
            zhi[q] = sz[2 * q + 1] - sz[2 * q];
        }
        M[0] = lo[0] + lo[1];
        M[1] = hi[0] + hi[1];
        M[2] = (lo[1] + ylo[1]) + (ylo[0] - lo[0]);
        M[3] = (hi[1] + yhi[1]) + (yhi[0] - hi[0]);
        Z[0] = zlo[0] + zlo[1];
        Z[1] = zhi[0] + zhi[1];
        Z[2] = zlo[1] - zlo[0];
        Z[3] = zhi[1] - zhi[0];
    }
    // along z with the lane of the other side: this lane ends with S without z (hz = 0) or with z (1)
    double r[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const double T = fma(hz ? 1.0 : -1.0, M[t], Z[t]);
        const double give = hz ? M[t] : T, keep = hz ? T : M[t];
        r[t] = keep + __shfl_xor_sync(0xffffffffu, give, 4);
    }
    // back to corners: r_c = sum_S sigma_{c,S} gamma^|S| M_S
    {
        const double a0 = fma(-gam, r[1], r[0]), a1 = fma(gam, r[1], r[0]), b0 = fma(-gam, r[3], r[2]), b1 = fma(gam, r[3], r[2]);
        r[0] = fma(-gam, b0, a0);
        r[1] = fma(-gam, b1, a1);
        r[2] = fma(gam, b0, a0);
        r[3] = fma(gam, b1, a1);
    }
    const double wq = A.lc[lv][6];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const double o = __shfl_xor_sync(0xffffffffu, r[t], 4);
        r[t] = wq * (hz ? fma(gam, r[t], o) : fma(-gam, o, r[t]));
        const int cr = t | (hz << 2);
        const int32_t ic = __shfl_sync(0xffffffffu, id, (lane & ~7) | cr);
        if (valid) {
            if (A.sv) ((double*)A.sv)[32 * idx + 4 * cr + k] = r[t];
            else scatter1(A, ic, k, r[t]);
        }
    }
    __syncwarp();   // the rows and the exchange area are rewritten by later elements
}

// One Out element on 8 lanes of a warp (lane & 7 = corner c): the element's rows `nd` are in
// shared memory (8 rows of CS, stride CS); the warp's moment rows s_mw [32][MSTR].  Thread c
// transforms column c of the rows into monomial coefficients, evaluates Gauss point c (monomials m),
// writes the point's 32 monomial moments, then sums moment column S = c over the 8 points and runs
// the backward butterfly: node c's rows, scattered (or stored to the element's slot).  Every lane of
// the warp takes part (valid: this lane's element exists).
// IL: with packed float duals, rewrite the rows with (value, tangent) interleaved so every 16-byte
// row load yields two dual pairs in place (off in the fused kernel, whose register budget it strains)
template <class T, bool JV, bool IL = (JV && sizeof(T) == 4)>
__device__ __forceinline__ void interior_element(const Args& A, T* nd, T* s_mw, const T m[8], int lane, int64_t idx,
                                                 bool valid, int lv, int prob, int32_t id) {
    typedef typename std::conditional<JV, Dual<T, sizeof(T) == 4>, T>::type S;
    constexpr int MSTR = IntShape<T>::MSTR;
    const int c = lane & 7;
    T* mrow = s_mw + lane * MSTR;
    const T* mcol = s_mw + (lane >> 3) * 8 * MSTR + 4 * c;
    __syncwarp();
    {   // corner values -> monomial coefficients: thread c transforms column c of the element's rows
        if constexpr (IL) {
            columns_to_monomial_interleaved<T>(nd, c);
        } else if (c < 7) {
            column_to_monomial<T>(nd + c);
            if (JV) column_to_monomial<T>(nd + CT + c);
        }
        if (A.ndf && c < 3) column_to_monomial<T>(nd + CF + c);
    }
    __syncwarp();
    const T g = lvl_g<T>(A, lv);
    const Phys<T> P(A, prob);
    S cf[16];
    vms_point_modal<S, T, IL>(A, P, m, nd, CS, g, cf);
    const T wq = lvl_w<T>(A, lv), wqg = wq * g;
    // F, G multiply phi; S, H multiply physical gradients = g x reference gradients
    T w16[16];
    for (int k = 0; k < 16; ++k) w16[k] = ((k < 3 || k == 12) ? wq : wqg) * Pick<T, JV>::get(cf[k]);
    T M[32];
    for (int k = 0; k < 32; ++k) M[k] = T(0);
    add_moments<T>(m, w16, M);
    for (int k = 0; k < 32; k += 4) st4s<T>(mrow + k, M[k], M[k + 1], M[k + 2], M[k + 3]);
    __syncwarp();
    T r[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        T v[4];
        ld4s<T>(mcol + q * MSTR, v);
        r[0] += v[0]; r[1] += v[1]; r[2] += v[2]; r[3] += v[3];
    }
    for (int k = 0; k < 4; ++k) r[k] = hadamard_bwd<1>(r[k], c);
    if (A.sv) {
        // deterministic scatter: node c's 4 rows into the element's slot (one 16- or 32-byte store)
        if (valid) st4s<T>((T*)A.sv + 32 * idx + 4 * c, r[0], r[1], r[2], r[3]);
    } else if constexpr (sizeof(T) == 4) {
        // corners of this warp's 4 elements that are the same node add their rows in shared memory
        // first; one lane per node scatters (fewer float64 atomics; float64: the plain scatter is faster)
        const unsigned grp = __match_any_sync(0xffffffffu, valid ? id : -1 - lane);
        __syncwarp();   // every lane has read its moment columns
        st4s<T>(mrow, r[0], r[1], r[2], r[3]);
        __syncwarp();
        if (valid && lane == __ffs(grp) - 1) {
            T t[4] = {T(0), T(0), T(0), T(0)};
            for (unsigned gm = grp; gm; gm &= gm - 1) {
                T v[4];
                ld4s<T>(s_mw + (__ffs(gm) - 1) * MSTR, v);
                for (int k = 0; k < 4; ++k) t[k] += v[k];
            }
            scatter_t(A, id, t);
        }
    } else {
        if (valid) scatter_t(A, id, r);
    }
    __syncwarp();   // the rows and the moments are rewritten by later elements
}

// Gauss point c of the 2x2x2 rule (xi_k = +-1/sqrt(3) by bit k of c) in monomial form
template <class T>
__device__ __forceinline__ void gauss_monomials(int c, T m[8]) {
    const T gauss = (T)0.57735026918962576451;
    T xi[3];
    for (int k = 0; k < 3; ++k) xi[k] = ((c >> k) & 1) ? gauss : -gauss;
    monomials<T>(xi, m);
}

// Persistent: a block walks element groups with a grid stride; while it computes group g its
// threads already stream the node rows of group g + stride into the other shared buffer
// (cp.async), so the gather latency hides behind the arithmetic.  Each warp computes 4 of the
// group's 16 elements (interior_element).
// MINB: resident blocks per SM the register allocation is made for (4: up to 128 registers per thread;
// 5: up to 102, a few spills, one more block of warps to hide latency with)
// GEN: float64 elements by the code of the float32 ones (see generic / GEN above)
template <class T, bool JV, int MINB = (sizeof(T) == 4 ? 4 : 2), bool GEN = false>
__global__ void __launch_bounds__(IntShape<T>::THREADS, MINB) vms_interior(Args A, const int32_t* __restrict__ oconn,
                                                    const uint8_t* __restrict__ olev,
                                                    const uint16_t* __restrict__ oprob, int64_t n) {
    constexpr int EPB = IntShape<T>::EPB, ESTR = IntShape<T>::ESTR, MSTR = IntShape<T>::MSTR;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* s_nd = reinterpret_cast<T*>(smem_raw);          // [2][EPB][ESTR]: 8 rows of CS per element
    T* s_m = s_nd + 2 * EPB * ESTR;                     // [EPB][8][MSTR]
    const int c = threadIdx.x & 7, le = threadIdx.x >> 3, lane = threadIdx.x & 31;
    const int64_t ngroups = (n + EPB - 1) / EPB;
    int64_t gi = blockIdx.x;
    if (A.skip && *A.skip) return;   // a captured solver step after its cycle ended
    if (gi >= ngroups) return;
    auto corner_id = [&](int64_t grp) -> int32_t {
        int64_t idx = grp * EPB + le;
        if (idx >= n) idx = n - 1;
        return __ldg(oconn + 8 * idx + c);
    };
    // level (and problem) of this lane's element of a group, loaded a group ahead of its use
    auto level_prob = [&](int64_t grp) -> int {
        int64_t idx = grp * EPB + le;
        if (idx >= n) idx = n - 1;
        return (int)__ldg(olev + idx) | (oprob ? (int)oprob[idx] << 8 : -256);
    };
    auto row = [&](int buf) -> T* { return s_nd + (buf * EPB + le) * ESTR + c * CS; };
    int32_t id_cur = corner_id(gi);
    corner_async<T, JV>(A, id_cur, row(0));
    cp_commit();
    int32_t id_next = gi + gridDim.x < ngroups ? corner_id(gi + gridDim.x) : 0;
    int lp_cur = level_prob(gi);
    T m[8];
    gauss_monomials<T>(c, m);
    T* s_mw = s_m + (threadIdx.x & ~31u) * MSTR;
    int buf = 0;
    for (; gi < ngroups; gi += gridDim.x) {
        const int64_t gnext = gi + gridDim.x;
        if (gnext < ngroups) corner_async<T, JV>(A, id_next, row(buf ^ 1));
        cp_commit();
        const int32_t id_after = gnext + gridDim.x < ngroups ? corner_id(gnext + gridDim.x) : 0;
        const int lp_next = gnext < ngroups ? level_prob(gnext) : 0;
        cp_wait<1>();
        const int64_t idx = gi * EPB + le;
        if constexpr (sizeof(T) == 8 && !GEN)
            interior_element64<JV>(A, s_nd + (buf * EPB + le) * ESTR, s_mw, lane, idx, idx < n, lp_cur & 255, lp_cur >> 8, id_cur);
        else
            interior_element<T, JV>(A, s_nd + (buf * EPB + le) * ESTR, s_mw, m, lane, idx, idx < n, lp_cur & 255,
                                    lp_cur >> 8, id_cur);
        id_cur = id_next;
        id_next = id_after;
        lp_cur = lp_next;
        buf ^= 1;
    }
    cp_wait<0>();
}

// ------------------------------------------------------------------------------------------
// Intercepted elements: one warp per element
// ------------------------------------------------------------------------------------------
constexpr int WPB = 4;   // warps per block of the per-element surface kernel

// Warp epilogue of the per-element kernels: lane l holds the monomial moments M of its points;
// sum them over the lanes (transpose through shared memory s_m [32][32 + pad]), run the backward
// butterfly so lane 4 a + k holds row (node a, component k), and scatter node a from lane 4 a.
// my_id: the node id of corner (lane & 7).
// extra: a float64 addend of this lane's row (node a = lane / 4, component lane % 4).  With the
// deterministic scatter the 32 rows go to a slot instead: vdst (element precision, volume terms)
// or sdst (float64, surface terms), row a * 4 + k at lane 4 a + k.
template <class T>
__device__ __forceinline__ void warp_scatter_moments(const Args& A, const T M[32], T* s_m, int lane, int32_t my_id,
                                                     double extra = 0.0, T* vdst = nullptr, double* sdst = nullptr) {
    constexpr int MSTR = 32 + 16 / (int)sizeof(T);
    T* mrow = s_m + lane * MSTR;
    for (int k = 0; k < 32; k += 4) st4s<T>(mrow + k, M[k], M[k + 1], M[k + 2], M[k + 3]);
    __syncwarp();
    T acc = T(0);
#pragma unroll 8
    for (int t = 0; t < 32; ++t) acc += s_m[t * MSTR + lane];
    acc = hadamard_bwd<4>(acc, lane >> 2);
    if (vdst) { vdst[lane] = acc; return; }
    const double row = (double)acc + extra;
    if (sdst) { sdst[lane] = row; return; }
    const int a = lane >> 2;
    double r[4];
    for (int k = 0; k < 4; ++k) r[k] = __shfl_sync(0xffffffffu, row, (lane & ~3) + k);
    const int32_t id = __shfl_sync(0xffffffffu, my_id, a);
    if ((lane & 3) == 0) scatter(A, id, r);
}

// One Intercepted element on one warp: lane l evaluates sub-cell points l, l + 32, ... and accumulates
// their monomial moments, summed over the lanes at the end (warp_scatter_moments).  s_nd [8 * CS] and
// s_m [32 * MSTR] are the warp's shared rows; idx the element's position in the list.
template <class T, bool JV>
__device__ __forceinline__ void cut_element(const Args& A, const int32_t* __restrict__ list, const int64_t* __restrict__ off,
                                            const void* __restrict__ pts, int64_t idx, T* s_nd, T* s_m, int lane) {
    typedef typename std::conditional<JV, Dual<T>, T>::type S;
    const int32_t e = list[idx];
    // every 8-lane group gathers the 8 corner rows and forms their monomial coefficients; lanes 0-7 store them
    const int c8 = lane & 7;
    const int32_t my_id = A.conn[8 * (int64_t)e + c8];
    {
        T rw[CS];
        corner_data<T, JV>(A, my_id, rw);
        for (int j = 0; j < 7; ++j) rw[j] = hadamard_fwd(rw[j], c8);
        if (JV)
            for (int j = 0; j < 7; ++j) rw[CT + j] = hadamard_fwd(rw[CT + j], c8);
        if (A.ndf)
            for (int j = 0; j < 3; ++j) rw[CF + j] = hadamard_fwd(rw[CF + j], c8);
        if (lane < 8)
            for (int j = 0; j < CS; ++j) s_nd[lane * CS + j] = rw[j];
    }
    __syncwarp();
    const T g = lvl_g<T>(A, A.lev[e]);
    const T det = lvl_w<T>(A, A.lev[e]);
    const Phys<T> P(A, prob_of(A, e));
    // lane l evaluates points q0 + l, q0 + l + 32, ... and accumulates their monomial moments
    T M[32];
    for (int k = 0; k < 32; ++k) M[k] = T(0);
    const int64_t q0 = off[idx], q1 = off[idx + 1];
    for (int64_t q = q0 + lane; q < q1; q += 32) {
        T pt[4];
        load_pt<T>(pts, q, pt);
        T m[8];
        monomials<T>(pt, m);
        S cf[16];
        vms_point_modal<S, T>(A, P, m, s_nd, CS, g, cf);
        const T wq = pt[3] * det, wqg = wq * g;
        T w16[16];
        for (int k = 0; k < 16; ++k) w16[k] = ((k < 3 || k == 12) ? wq : wqg) * Pick<T, JV>::get(cf[k]);
        add_moments<T>(m, w16, M);
    }
    warp_scatter_moments<T>(A, M, s_m, lane, my_id, 0.0, A.sv ? (T*)A.sv + 32 * (A.n_out_slots + idx) : nullptr);
}

// The same element, with the same sums, on a block of four warps: each warp evaluates every fourth round of
// 32 points and leaves the coefficients in shared memory, then takes one component's moments of all four
// rounds in order (lane l: points l, l + 32, ...).  Where there are few elements, the longest of them (a
// thousand points and more on one warp) is the kernel's time: 7.3 k element sphere, 776 elements, mixed J v
// 23 -> 15 us; float64 (the generic code of mixed solves, bound by the FP64 pipe of the SMs that got the long
// elements) R 480 -> 241, J v 746 -> 368 us.  With many elements the two barriers per 128 points cost more
// than they give: float32 meshes of more than kSplitCut elements per SM keep a warp per element.
constexpr int kSplitCut = 16;
template <class T, bool JV>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 4 : 2) vms_cut_split(Args A, const int32_t* __restrict__ list,
                                                                            const int64_t* __restrict__ off,
                                                                            const void* __restrict__ pts,
                                                                            const int32_t* __restrict__ order) {
    typedef typename std::conditional<JV, Dual<T>, T>::type S;
    constexpr int MSTR = 32 + 16 / (int)sizeof(T);
    __shared__ __align__(16) T s_nd[8 * CS];
    __shared__ __align__(16) T s_m[32 * MSTR];
    __shared__ T s_w[4][16][33], s_x[4][3][33];
    if (A.skip && *A.skip) return;   // a captured solver step after its cycle ended
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t idx = order ? (int64_t)order[blockIdx.x] : blockIdx.x;
    const int32_t e = list[idx];
    const int c8 = lane & 7;
    const int32_t my_id = A.conn[8 * (int64_t)e + c8];
    if (w == 0) {
        T rw[CS];
        corner_data<T, JV>(A, my_id, rw);
        for (int j = 0; j < 7; ++j) rw[j] = hadamard_fwd(rw[j], c8);
        if (JV)
            for (int j = 0; j < 7; ++j) rw[CT + j] = hadamard_fwd(rw[CT + j], c8);
        if (A.ndf)
            for (int j = 0; j < 3; ++j) rw[CF + j] = hadamard_fwd(rw[CF + j], c8);
        if (lane < 8)
            for (int j = 0; j < CS; ++j) s_nd[lane * CS + j] = rw[j];
    }
    __syncthreads();
    const T g = lvl_g<T>(A, A.lev[e]);
    const T det = lvl_w<T>(A, A.lev[e]);
    const Phys<T> P(A, prob_of(A, e));
    T M[8];   // component w
    for (int k = 0; k < 8; ++k) M[k] = T(0);
    const int64_t q0 = off[idx], q1 = off[idx + 1];
    for (int64_t base = q0; base < q1; base += 128) {
        const int64_t q = base + 32 * w + lane;
        if (q < q1) {
            T pt[4];
            load_pt<T>(pts, q, pt);
            T m[8];
            monomials<T>(pt, m);
            S cf[16];
            vms_point_modal<S, T>(A, P, m, s_nd, CS, g, cf);
            const T wq = pt[3] * det, wqg = wq * g;
            for (int k = 0; k < 16; ++k) s_w[w][k][lane] = ((k < 3 || k == 12) ? wq : wqg) * Pick<T, JV>::get(cf[k]);
            for (int k = 0; k < 3; ++k) s_x[w][k][lane] = pt[k];
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (base + 32 * r + lane < q1) {
                const T xi[3] = {s_x[r][0][lane], s_x[r][1][lane], s_x[r][2][lane]};
                T m[8];
                monomials<T>(xi, m);
                const T f = s_w[r][w < 3 ? w : 12][lane], sx = s_w[r][w < 3 ? 3 + 3 * w : 13][lane],
                        sy = s_w[r][w < 3 ? 4 + 3 * w : 14][lane], sz = s_w[r][w < 3 ? 5 + 3 * w : 15][lane];
                auto add = [&](int Sx, T s, T x) { M[Sx] = fma(s, x, M[Sx]); };   // as add_moments
                add(0, m[0], f);
                add(1, m[1], f); add(1, m[0], sx);
                add(2, m[2], f); add(2, m[0], sy);
                add(3, m[3], f); add(3, m[2], sx); add(3, m[1], sy);
                add(4, m[4], f); add(4, m[0], sz);
                add(5, m[5], f); add(5, m[4], sx); add(5, m[1], sz);
                add(6, m[6], f); add(6, m[4], sy); add(6, m[2], sz);
                add(7, m[7], f); add(7, m[6], sx); add(7, m[5], sy); add(7, m[3], sz);
            }
        __syncthreads();
    }
    for (int k = 0; k < 8; ++k) s_m[lane * MSTR + 4 * k + w] = M[k];
    __syncthreads();
    if (w > 0) return;
    T row[32];
    for (int k = 0; k < 32; k += 4) ld4s<T>(&s_m[lane * MSTR + k], row + k);
    __syncwarp();
    warp_scatter_moments<T>(A, row, s_m, lane, my_id, 0.0, A.sv ? (T*)A.sv + 32 * (A.n_out_slots + idx) : nullptr);
}

// ------------------------------------------------------------------------------------------
// Intercepted elements in float64 (see Const64: FP64 instructions are the cost).  Per point the fields
// come from the Hadamard coefficients by Horner steps along x, y, z, whose intermediates are the
// gradients and mixed derivatives (11 or 12 multiply-adds per column; monomial by monomial 22), and the
// 32 moments take the transposed steps (16 per component; 20 before).  An element's points are dealt
// to four parts (part p: points 32 p + lane, + 128, ...) that different warps take, so the longest
// element (8^(L_max + 1) points) is not one warp's serial work; each part sums its lanes, the parts are
// added in order.  The fused kernel runs the same four parts on one warp: the same bits.
//   7.3 k element sphere (234 k points in 776 elements), one R and one J v: 1.44 -> 0.53 ms.
// ------------------------------------------------------------------------------------------
constexpr int kCutParts = 4, kCutCols = 14;   // columns: 7 values, 4 tangents (u_s, p), 3 force

// coefficient columns of element e, [column][8], by a block or warp of nt threads (a multiple of 32)
template <bool JV>
__device__ __forceinline__ void cut_columns64(const Args& A, int32_t e, double* s_col, int t0, int nt) {
    for (int t = t0; t < 8 * kCutCols + 16; t += nt) {   // 4 x 32: whole warps (the shuffles)
        const int col = t >> 3, c = t & 7;
        const int64_t id = A.conn[8 * (int64_t)e + c];
        double x = 0.0;
        if (col < 7) x = __ldg((const double*)A.ndv + 8 * id + col);
        else if (col < 11) { if (JV) x = __ldg((const double*)A.ndt + 8 * id + col - 7); }
        else if (col < 14) { if (A.ndf) x = __ldg((const double*)A.ndf + 4 * id + col - 11); }
        x = hadamard_fwd(x, c);
        if (col < kCutCols) s_col[t] = x;
    }
}

// lane's sum of moment row `lane` (4 S + k) over part p's points of the element, points [q0, q1)
template <bool JV>
__device__ __forceinline__ double cut_part64(const Args& A, const Const64& C, double det, const double* s_col,
                                             const double* __restrict__ pts, int64_t q0, int64_t q1, int p, double* s_m, int lane) {
    constexpr int MSTR = 34;
    const int64_t first = q0 + 32 * p;
    if (first >= q1) return 0.0;
    double M[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) M[k] = 0.0;
    for (int64_t q = first + lane; q < q1; q += 32 * kCutParts) {
        double pt[4];
        load_pt<double>(pts, q, pt);
        const double x = pt[0], y = pt[1], z = pt[2];
        Point64 F;
        Tangent64 D;
        auto value = [&](int col) {
            const double* a = s_col + 8 * col;
            const double b0 = fma(x, a[1], a[0]), b1 = fma(x, a[3], a[2]), b2 = fma(x, a[5], a[4]), b3 = fma(x, a[7], a[6]);
            return fma(z, fma(y, b3, b2), fma(y, b1, b0));
        };
        // value, gradient and mixed second derivatives (xy, xz, yz)
        auto all = [&](int col, double& v, double g[3], double m[3]) {
            const double* a = s_col + 8 * col;
            const double b0 = fma(x, a[1], a[0]), b1 = fma(x, a[3], a[2]), b2 = fma(x, a[5], a[4]), b3 = fma(x, a[7], a[6]);
            const double c1 = fma(y, b3, b2), j = fma(y, a[7], a[5]);
            v = fma(z, c1, fma(y, b1, b0));
            g[2] = c1;
            g[1] = fma(z, b3, b1);
            g[0] = fma(z, j, fma(y, a[3], a[1]));
            m[0] = fma(z, a[7], a[3]);
            m[1] = j;
            m[2] = b3;
        };
        {
            double m[3][3], unused[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) all(i, F.u[i], F.G[i], m[i]);
            F.H[0] = m[1][0] + m[2][1];
            F.H[1] = m[0][0] + m[2][2];
            F.H[2] = m[0][1] + m[1][2];
            all(3, F.p, F.gp, unused);
#pragma unroll
            for (int i = 0; i < 3; ++i) F.a[i] = value(4 + i);
            if (A.ndf)
                for (int i = 0; i < 3; ++i) F.f[i] = value(11 + i);
            if (JV) {
#pragma unroll
                for (int i = 0; i < 3; ++i) all(7 + i, D.u[i], D.G[i], m[i]);
                D.H[0] = m[1][0] + m[2][1];
                D.H[1] = m[0][0] + m[2][2];
                D.H[2] = m[0][1] + m[1][2];
                all(10, D.p, D.gp, unused);
            }
        }
        double W[16];
        pointwise64<JV>(C, A.ndf != nullptr, A.c0th, F, D, W);
        const double w = pt[3] * det, yz = y * z;
#pragma unroll
        for (int k = 0; k < 16; ++k) W[k] *= w;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double f = W[k], sx = W[4 + 3 * k], sy = W[5 + 3 * k], sz = W[6 + 3 * k];
            const double c = fma(z, f, sz), b = fma(y, f, sy), d = fma(y, c, z * sy);
            M[k] += f;
            M[4 + k] = fma(x, f, M[4 + k] + sx);
            M[8 + k] += b;
            M[12 + k] = fma(x, b, fma(y, sx, M[12 + k]));
            M[16 + k] += c;
            M[20 + k] = fma(x, c, fma(z, sx, M[20 + k]));
            M[24 + k] += d;
            M[28 + k] = fma(x, d, fma(yz, sx, M[28 + k]));
        }
    }
    const int rows = (int)min((int64_t)32, q1 - first);   // lanes that had a point
    double* mrow = s_m + lane * MSTR;
#pragma unroll
    for (int k = 0; k < 32; k += 2) *reinterpret_cast<double2*>(mrow + k) = make_double2(M[k], M[k + 1]);
    __syncwarp();
    double acc = s_m[lane];
    for (int t = 1; t < rows; ++t) acc += s_m[t * MSTR + lane];
    __syncwarp();
    return acc;
}

// rows of the element from the summed moments (lane 4 a + k: node a, component k) to its slot or the nodes
__device__ __forceinline__ void cut_rows64(const Args& A, int32_t e, int64_t idx, double acc, int lane) {
    acc = hadamard_bwd<4>(acc, lane >> 2);
    if (A.sv) ((double*)A.sv)[32 * (A.n_out_slots + idx) + lane] = acc;
    else scatter1(A, A.conn[8 * (int64_t)e + (lane >> 2)], lane & 3, acc);
}

__device__ __forceinline__ int cut_parts(int64_t points) { return (int)min((int64_t)kCutParts, (points + 31) / 32); }

// a block of W warps per element (warp w: parts w, w + W, ...)
template <bool JV, int W>
__global__ void __launch_bounds__(32 * W, 8 / W) vms_cut64(Args A, const int32_t* __restrict__ list, const int64_t* __restrict__ off,
                                                          const double* __restrict__ pts, const int32_t* __restrict__ order) {
    __shared__ __align__(16) double s_col[8 * kCutCols], s_m[W][32 * 34], s_part[kCutParts][32];
    if (A.skip && *A.skip) return;   // a captured solver step after its cycle ended
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t idx = order ? (int64_t)order[blockIdx.x] : blockIdx.x;
    const int32_t e = list[idx];
    cut_columns64<JV>(A, e, s_col, threadIdx.x, 32 * W);
    const int64_t q0 = off[idx], q1 = off[idx + 1];
    const int lv = A.lev[e];
    const Const64 C(A, Phys<double>(A, prob_of(A, e)), lv, A.lc[lv][0], A.lc[lv][1]);
    __syncthreads();
    for (int p = w; p < kCutParts; p += W) s_part[p][lane] = cut_part64<JV>(A, C, A.lc[lv][6], s_col, pts, q0, q1, p, s_m[w], lane);
    __syncthreads();
    if (w > 0) return;
    double acc = s_part[0][lane];
    for (int p = 1, np = cut_parts(q1 - q0); p < np; ++p) acc += s_part[p][lane];
    cut_rows64(A, e, idx, acc, lane);
}

// the same element on one warp (fused kernel); s: 8 kCutCols + 32 x 34 doubles of the warp
template <bool JV>
__device__ __forceinline__ void cut_element64(const Args& A, const int32_t* __restrict__ list, const int64_t* __restrict__ off,
                                              const double* __restrict__ pts, int64_t idx, double* s, int lane) {
    const int32_t e = list[idx];
    cut_columns64<JV>(A, e, s, lane, 32);
    const int64_t q0 = off[idx], q1 = off[idx + 1];
    const int lv = A.lev[e];
    const Const64 C(A, Phys<double>(A, prob_of(A, e)), lv, A.lc[lv][0], A.lc[lv][1]);
    __syncwarp();
    double acc = 0.0;
    for (int p = 0, np = cut_parts(q1 - q0); p < np; ++p) {
        const double x = cut_part64<JV>(A, C, A.lc[lv][6], s, pts, q0, q1, p, s + 8 * kCutCols, lane);
        acc = p == 0 ? x : acc + x;
    }
    cut_rows64(A, e, idx, acc, lane);
}

// float32: W warps per block (a tile shape the autotuner picks); `order` (or null) permutes the list
template <bool JV, int W>
__global__ void __launch_bounds__(32 * W, 16 / W) vms_cut(Args A, const int32_t* __restrict__ list,
                                                    const int64_t* __restrict__ off, const void* __restrict__ pts,
                                                    const int32_t* __restrict__ order, int64_t n) {
    constexpr int MSTR = 36;
    __shared__ __align__(16) float s_nd[W][8 * CS];
    __shared__ __align__(16) float s_m[W][32 * MSTR];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t slot = (int64_t)blockIdx.x * W + w;
    if (A.skip && *A.skip) return;   // a captured solver step after its cycle ended
    if (slot >= n) return;
    cut_element<float, JV>(A, list, off, pts, order ? (int64_t)order[slot] : slot, &s_nd[w][0], &s_m[w][0], lane);
}

// ------------------------------------------------------------------------------------------
// Nitsche surface terms (Eq. weakbc), one thread per surface point: elements hosting few points
// ------------------------------------------------------------------------------------------
template <class T, bool JV>
__device__ __forceinline__ void surface_point(const Args& A, const int32_t* __restrict__ el, const double* __restrict__ xr,
                                              const double* __restrict__ nr, const double* __restrict__ wr, int64_t i) {
    typedef typename std::conditional<JV, Dual<T>, T>::type S;
    NitschePoint<S, T> P;
    const int32_t e = el[i];
    nitsche_fields<S, T, JV, false>(A, e, i, xr + 3 * i, nr + 3 * i, P);
    const T w = (T)wr[i];
    // (the penalty is added per element in float64 by nitsche_penalty)
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        S t[4];
        nitsche_rows<S, T, false>(A, P, c, T(0), t);
        double r[4];
        for (int k = 0; k < 4; ++k) r[k] = (double)(w * Pick<T, JV>::get(t[k]));
        if (A.ss) {
            double* d = A.ss + 32 * (A.n_dense_slots + i) + 4 * c;
            reinterpret_cast<double2*>(d)[0] = make_double2(r[0], r[1]);
            reinterpret_cast<double2*>(d)[1] = make_double2(r[2], r[3]);
        } else {
            scatter(A, P.ids[c], r);
        }
    }
}

template <class T, bool JV>
__global__ void __launch_bounds__(128) nitsche(Args A, const int32_t* __restrict__ el, const double* __restrict__ xr,
                                               const double* __restrict__ nr, const double* __restrict__ wr,
                                               const double* __restrict__ taub, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (A.skip && *A.skip) return;   // a captured solver step after its cycle ended
    surface_point<T, JV>(A, el, xr, nr, wr, i);
}

// ------------------------------------------------------------------------------------------
// Nitsche surface terms (Eq. weakbc), one warp per element hosting many surface points; lane l takes
// points l, l + 32, ... of the element.  Per point the 4 rows of corner c are
//   t_k = phi_c [tau_B d_k - tr_k - [u.n < 0] rho (u.n) d_k] - mu g sum_j d_j phi_c (n_j d_k + n_k d_j),
//   t_p = -phi_c (d.n),   d = u_s - g, tr = -p n + 2 mu eps(u) n,
// i.e. coefficients of phi_c and of its reference gradient, accumulated as monomial moments.
// ------------------------------------------------------------------------------------------
template <class T, bool JV>
__device__ __forceinline__ void surface_element(const Args& A, const int32_t* __restrict__ list, const int64_t* __restrict__ off,
                                                const double* __restrict__ xr, const double* __restrict__ nr,
                                                const double* __restrict__ wr, int64_t idx, T* s_nd, T* s_m, int lane) {
    typedef typename std::conditional<JV, Dual<T>, T>::type S;
    const int32_t e = list[idx];
    // corner rows: u_s (0-2), p (3), jump d = u_s - g_body formed in float64 (4-6), tangents at CT
    // (the penalty is added per element in float64 by nitsche_penalty)
    const int c8 = lane & 7;
    const int32_t my_id = A.conn[8 * (int64_t)e + c8];
    {
        T a8[8], t8[8] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
        ld8<T>(A.ndv, my_id, a8);
        if (JV) ld8<T>(A.ndt, my_id, t8);
        double u4[4], up4[4];
        gather(A, A.U, my_id, u4);
        if (!A.theta1) gather(A, A.Up, my_id, up4);
        T rw[CS];
        for (int k = 0; k < 3; ++k) {
            const double usk = A.theta1 ? u4[k] : A.theta * u4[k] + (1.0 - A.theta) * up4[k];
            rw[k] = a8[k];
            rw[4 + k] = (T)(usk - A.g[k]);
            rw[CT + k] = t8[k];
            rw[CT + 4 + k] = t8[k];
        }
        rw[3] = a8[3];
        rw[CT + 3] = t8[3];
        for (int j = 0; j < 7; ++j) rw[j] = hadamard_fwd(rw[j], c8);
        if (JV)
            for (int j = 0; j < 7; ++j) rw[CT + j] = hadamard_fwd(rw[CT + j], c8);
        if (lane < 8) {
            for (int j = 0; j < 7; ++j) s_nd[lane * CS + j] = rw[j];
            if (JV)
                for (int j = 0; j < 7; ++j) s_nd[lane * CS + CT + j] = rw[CT + j];
        }
    }
    __syncwarp();
    const T g = lvl_g<T>(A, A.lev[e]);
    T mu, rho;
    {
        const Phys<T> Ph(A, prob_of(A, e));
        mu = Ph.mu;
        rho = Ph.rho;
    }
    T M[32];
    for (int k = 0; k < 32; ++k) M[k] = T(0);
    const int64_t q0 = off[idx], q1 = off[idx + 1];
    for (int64_t q = q0 + lane; q < q1; q += 32) {
        T xi[3], nn[3], m[8];
        for (int k = 0; k < 3; ++k) { xi[k] = (T)xr[3 * q + k]; nn[k] = (T)nr[3 * q + k]; }
        // the jump relative to g_body at the corners, corrected to this point's g (its value enters
        // the tangent of the inflow term)
        T dg[3] = {T(0), T(0), T(0)};
        if (A.gpts) {
            const double* gq = point_g(A, q);
            for (int k = 0; k < 3; ++k) dg[k] = (T)(A.g[k] - gq[k]);
        }
        monomials<T>(xi, m);
        // u_s, grad u_s, p, d at the point
        S us[3], Gu[3][3], p, d[3];
        for (int i = 0; i < 3; ++i) { us[i] = zero<S>(); d[i] = zero<S>(); for (int j = 0; j < 3; ++j) Gu[i][j] = zero<S>(); }
        p = zero<S>();
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const T* r = &s_nd[t * CS];
            S a[7];
            for (int j = 0; j < 7; ++j) a[j] = make<S, T>(r[j], JV ? r[CT + j] : T(0));
            for (int i = 0; i < 3; ++i) {
                us[i] = madd(m[t], a[i], us[i]);
                d[i] = madd(m[t], a[4 + i], d[i]);
            }
            p = madd(m[t], a[3], p);
            for (int k = 0; k < 3; ++k)
                if (t & (1 << k))
                    for (int i = 0; i < 3; ++i) Gu[i][k] = madd(m[t ^ (1 << k)], a[i], Gu[i][k]);
        }
        for (int i = 0; i < 3; ++i) {
            d[i] = d[i] + dg[i];
            for (int j = 0; j < 3; ++j) Gu[i][j] = g * Gu[i][j];
        }
        const S un = mmadd(us[2], S(make<S, T>(nn[2], T(0))), mmadd(us[1], S(make<S, T>(nn[1], T(0))), us[0] * nn[0]));
        const S dn = madd(nn[2], d[2], madd(nn[1], d[1], nn[0] * d[0]));
        const bool inflow = value(un) < T(0);
        const T wq = (T)wr[q], wqg = wq * g;
        T c[16];
        for (int k = 0; k < 3; ++k) {
            S tr = (-nn[k]) * p;
            for (int j = 0; j < 3; ++j) tr = madd(mu * nn[j], Gu[k][j] + Gu[j][k], tr);
            S fk = T(-1) * tr;
            if (inflow) fk = fk - rho * (un * d[k]);
            c[k] = wq * Pick<T, JV>::get(fk);
            for (int j = 0; j < 3; ++j) c[3 + 3 * k + j] = (-wqg * mu) * Pick<T, JV>::get(madd(nn[j], d[k], nn[k] * d[j]));
        }
        c[12] = -wq * Pick<T, JV>::get(dn);
        c[13] = c[14] = c[15] = T(0);
        add_moments<T>(m, c, M);
    }
    warp_scatter_moments<T>(A, M, s_m, lane, my_id, 0.0, nullptr, A.ss ? A.ss + 32 * idx : nullptr);
}

template <class T, bool JV>
__global__ void __launch_bounds__(32 * WPB, sizeof(T) == 4 ? 2 : 1) nitsche_el(Args A, const int32_t* __restrict__ list,
                                                    const int64_t* __restrict__ off, const double* __restrict__ xr,
                                                    const double* __restrict__ nr, const double* __restrict__ wr,
                                                    const double* __restrict__ taub, int64_t n) {
    constexpr int PAD = 16 / (int)sizeof(T), MSTR = 32 + PAD;
    __shared__ __align__(16) T s_nd[WPB][8 * CS];
    __shared__ __align__(16) T s_m[WPB][32 * MSTR];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t idx = (int64_t)blockIdx.x * WPB + w;
    if (A.skip && *A.skip) return;   // a captured solver step after its cycle ended
    if (idx >= n) return;
    surface_element<T, JV>(A, list, off, xr, nr, wr, idx, &s_nd[w][0], &s_m[w][0], lane);
}

// ------------------------------------------------------------------------------------------
// One persistent launch over the volume quadrature buckets.  Every warp drains a device work queue
// on its own: first the Intercepted elements (8 .. 4096 sub-cell points), one per claim, longest
// first (the cost model of Eq. Wpart: a warp's time grows with its rounds of 32 points); then the
// Out elements, 4 per warp item, kFusedChunk items per claim, with their node rows double-buffered
// by cp.async as in vms_interior.  Longest items first, then small uniform ones, keeps every SM
// busy to the end whatever the mix (one mesh or many problems of a batch).  The surface terms run
// as their own kernels beside this one (their register budget would spill in it).
// ------------------------------------------------------------------------------------------
constexpr int kFusedWarps = 4;   // warps per block
constexpr int kFusedChunk = 8;   // Out warp items per claim

struct FusedQueue {
    const uint32_t* items;       // Intercepted-list positions, by decreasing point count
    int64_t n_items;
    unsigned long long* cnt;     // [3] claimed items, claimed Out warp items, finished blocks (zero at launch)
    const int32_t* oconn;
    const uint8_t* olev;
    const uint16_t* oprob;
    int64_t n_out;
    const int32_t* cut_list;
    const int64_t* cut_off;
    const void* cut_pts;
    int heavy_warps;             // warps per block that take the costly items before the Out elements
};

template <class T> struct FusedShape {
    static constexpr int ESTR = IntShape<T>::ESTR, MSTR = IntShape<T>::MSTR;
    // per warp: the Out layout (2 buffers x 4 elements of rows, 32 moment rows); the per-element
    // layouts (8 rows, 32 moment rows) fit inside it
    static constexpr int WARP = 2 * 4 * ESTR + 32 * MSTR;
    static_assert(8 * CS + 32 * MSTR <= WARP && 8 * kCutCols + 32 * 34 <= WARP, "per-element layout");
    static_assert((WARP * sizeof(T)) % 16 == 0 && (8 * CS * sizeof(T)) % 16 == 0, "16-byte rows");
    static constexpr size_t smem = (size_t)kFusedWarps * WARP * sizeof(T);
};

// GEN: as in vms_interior
template <class T, bool JV, bool GEN = false>
__global__ void __launch_bounds__(32 * kFusedWarps, sizeof(T) == 4 ? 4 : 2) vms_fused(Args A, FusedQueue Q) {
    constexpr int ESTR = FusedShape<T>::ESTR, MSTR = FusedShape<T>::MSTR;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    T* base = reinterpret_cast<T*>(smem_raw) + (threadIdx.x >> 5) * FusedShape<T>::WARP;
    if (A.skip && *A.skip) return;   // a captured solver step after its cycle ended
    // the costly items, one per claim
    auto drain_costly = [&]() {
        for (;;) {
            unsigned long long h = 0;
            if (lane == 0) h = atomicAdd(Q.cnt, 1ull);
            h = __shfl_sync(0xffffffffu, h, 0);
            if ((int64_t)h >= Q.n_items) break;
            if constexpr (sizeof(T) == 8 && !GEN)
                cut_element64<JV>(A, Q.cut_list, Q.cut_off, (const double*)Q.cut_pts, (int64_t)Q.items[h], base, lane);
            else
                cut_element<T, JV>(A, Q.cut_list, Q.cut_off, Q.cut_pts, (int64_t)Q.items[h], base, base + 8 * CS, lane);
            __syncwarp();   // the shared rows are reused by the next item
        }
    };
    // 1. the first heavy_warps warps of every block start on the costly items (the others go straight
    //    to the Out elements, so latency-bound costly work shares each SM with arithmetic-bound Out work)
    const bool heavy_first = (int)(threadIdx.x >> 5) < Q.heavy_warps;
    // 2. Out elements
    auto drain_out = [&]() {
        if (Q.n_out > 0) {
            const int c = lane & 7, le = lane >> 3;
            const int64_t n_wi = (Q.n_out + 3) / 4;
            int64_t pos = 0, end = 0;
            bool more = true;
            auto claim = [&]() -> int64_t {   // warp-uniform
                if (pos < end) return pos++;
                if (!more) return -1;
                unsigned long long b = 0;
                if (lane == 0) b = atomicAdd(Q.cnt + 1, (unsigned long long)kFusedChunk);
                b = __shfl_sync(0xffffffffu, b, 0);
                if ((int64_t)b >= n_wi) { more = false; return -1; }
                pos = (int64_t)b + 1;
                end = (int64_t)b + kFusedChunk < n_wi ? (int64_t)b + kFusedChunk : n_wi;
                return (int64_t)b;
            };
            auto corner_id = [&](int64_t wi) -> int32_t {
                int64_t idx = 4 * wi + le;
                if (idx >= Q.n_out) idx = Q.n_out - 1;
                return __ldg(Q.oconn + 8 * idx + c);
            };
            auto level_prob = [&](int64_t wi) -> int {   // loaded an item ahead of its use
                int64_t idx = 4 * wi + le;
                if (idx >= Q.n_out) idx = Q.n_out - 1;
                return (int)__ldg(Q.olev + idx) | (Q.oprob ? (int)Q.oprob[idx] << 8 : -256);
            };
            auto row = [&](int buf) -> T* { return base + (buf * 4 + le) * ESTR + c * CS; };
            T* s_mw = base + 8 * ESTR;
            int64_t cur = claim();
            if (cur >= 0) {
                T m[8];
                gauss_monomials<T>(c, m);
                int32_t id_cur = corner_id(cur);
                corner_async<T, JV>(A, id_cur, row(0));
                cp_commit();
                int lp_cur = level_prob(cur);
                int64_t nxt = claim();
                int32_t id_next = nxt >= 0 ? corner_id(nxt) : 0;
                int buf = 0;
                while (cur >= 0) {
                    if (nxt >= 0) corner_async<T, JV>(A, id_next, row(buf ^ 1));
                    cp_commit();
                    const int64_t aft = nxt >= 0 ? claim() : -1;
                    const int32_t id_after = aft >= 0 ? corner_id(aft) : 0;
                    const int lp_next = nxt >= 0 ? level_prob(nxt) : 0;
                    cp_wait<1>();
                    const int64_t idx = 4 * cur + le;
                    if constexpr (sizeof(T) == 8 && !GEN)
                        interior_element64<JV>(A, base + (buf * 4 + le) * ESTR, s_mw, lane, idx, idx < Q.n_out, lp_cur & 255,
                                               lp_cur >> 8, id_cur);
                    else
                        interior_element<T, JV>(A, base + (buf * 4 + le) * ESTR, s_mw, m, lane, idx, idx < Q.n_out,
                                                lp_cur & 255, lp_cur >> 8, id_cur);
                    cur = nxt;
                    nxt = aft;
                    id_cur = id_next;
                    id_next = id_after;
                    lp_cur = lp_next;
                    buf ^= 1;
                }
                cp_wait<0>();
            }
        }
    };
    // one call site each (the bodies are inlined once): costly items then Out elements, or the reverse
    for (int phase = 0; phase < 2; ++phase) {
        if ((phase == 0) == heavy_first) drain_costly();
        else drain_out();
    }
    // 3. the last block to finish zeroes the counters for the next launch (every claim of every block
    //    precedes its count here)
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(Q.cnt + 2, 1ull) == (unsigned long long)gridDim.x - 1) {
            Q.cnt[0] = 0;
            Q.cnt[1] = 0;
            Q.cnt[2] = 0;
            __threadfence();
        }
    }
}

// ------------------------------------------------------------------------------------------
// Nitsche penalty in float64, one thread per surface-hosting element.  Over the element's surface
// points the penalty rows are linear in the corner values with a matrix that does not depend on the
// state,
//   r_{a,k} = sum_q w_q tau_B(q) phi_a(x_q) (u_s(x_q) - g(x_q))_k
//           = C_b mu sum_b Pen_ab (u_s,b - g_body)_k + C_b mu sum_q (w_q / h_b) phi_a (g_body - g_q)_k,
//   Pen_ab = sum_q (w_q / h_b) phi_a(x_q) phi_b(x_q)      (float64, built with the mesh),
// so each call costs one 8 x 8 x 3 product per element instead of float64 work per point (the second
// sum only with per-point velocities).  J v: the tangent theta v in place of u_s - g_body.  The rows
// go to the element's surface slot (dense bucket) or to the slot of its first point (sparse bucket),
// after the surface kernel wrote it, or by float64 atomics.
// ------------------------------------------------------------------------------------------
template <bool JV>
__global__ void __launch_bounds__(128) nitsche_penalty(Args A, const int32_t* __restrict__ pe,
                                                       const int64_t* __restrict__ pslot,
                                                       const double* __restrict__ pen, int64_t n) {
    // eight threads per element: thread c fetches corner c's jump, then forms row c
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i = t >> 3;
    const int c = (int)(t & 7);
    if (A.skip && *A.skip) return;   // a captured solver step after its cycle ended (uniform over the grid)
    const bool live = i < n;
    const int64_t ii = live ? i : n - 1;
    const int32_t e = pe[ii];
    const double cbmu = A.Cb * Phys<double>(A, prob_of(A, e)).mu;
    const int32_t id = A.conn[8 * (int64_t)e + c];
    double dc[3];
    if (JV) {
        double v4[4];
        gather(A, A.V, id, v4);
        for (int k = 0; k < 3; ++k) dc[k] = A.theta * v4[k];
    } else {
        double u4[4], up4[4];
        gather(A, A.U, id, u4);
        if (!A.theta1) gather(A, A.Up, id, up4);
        for (int k = 0; k < 3; ++k) dc[k] = (A.theta1 ? u4[k] : A.theta * u4[k] + (1.0 - A.theta) * up4[k]) - A.g[k];
    }
    const double* P = pen + 36 * ii;   // upper triangle, row by row: (a, b >= a) at a * 8 - a (a - 1) / 2 + b - a
    double r[3] = {0.0, 0.0, 0.0};
    const unsigned base = threadIdx.x & 31 & ~7u;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const int lo = c < b ? c : b, hi = c < b ? b : c;
        const double m = cbmu * P[lo * 8 - lo * (lo - 1) / 2 + hi - lo];
        for (int k = 0; k < 3; ++k) r[k] = fma(m, __shfl_sync(0xffffffffu, dc[k], base | b), r[k]);
    }
    if (!live) return;
    if (A.ss) {
        double* dst = A.ss + 32 * pslot[i] + 4 * c;
        for (int k = 0; k < 3; ++k) dst[k] += r[k];
    } else {
        const double rr[4] = {r[0], r[1], r[2], 0.0};
        scatter(A, id, rr);
    }
}

// The residual's penalty with a velocity per surface point (the second sum above too): a warp per
// element, a lane per point.  Bound by the latency of the point data (two dependent loads, position
// then velocity) and by the narrow FP64 pipe, so every point is read and its basis formed once, by one
// lane, not by the eight threads of a corner in turn: 24 sums per lane, then halved over the lanes
// (27 additions) until lane 4 c + k holds row (c, k).  41 k element truck pair, 19,898 points:
// the residual with a velocity per point went from 325 to 81 us (this sum was 269 of them).
__global__ void __launch_bounds__(128) nitsche_penalty_points(Args A, const int32_t* __restrict__ pe,
                                                              const int64_t* __restrict__ pq,
                                                              const int64_t* __restrict__ pslot,
                                                              const double* __restrict__ pen, const double* __restrict__ xr,
                                                              const double* __restrict__ wr, const double* __restrict__ taub,
                                                              int64_t n) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;              // uniform over the warp
    if (A.skip && *A.skip) return;   // a captured solver step after its cycle ended
    const int lane = threadIdx.x & 31, c = lane >> 2, k = lane & 3;
    const int32_t e = pe[i];
    const double cbmu = A.Cb * Phys<double>(A, prob_of(A, e)).mu;
    const int32_t id = A.conn[8 * (int64_t)e + c];
    // component k of corner c's u_s - g_body (k = 3: unused)
    double u4[4], up4[4];
    gather(A, A.U, id, u4);
    if (!A.theta1) gather(A, A.Up, id, up4);
    double dc = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j)
        if (k == j) dc = (A.theta1 ? u4[j] : A.theta * u4[j] + (1.0 - A.theta) * up4[j]) - A.g[j];
    double s[24];   // [corner][component] of this lane's points
#pragma unroll
    for (int j = 0; j < 24; ++j) s[j] = 0.0;
    for (int64_t q = pq[i] + lane, q1 = pq[i + 1]; q < q1; q += 32) {
        const double* gq = point_g(A, q);
        double phi[8], t[3];
        basis_values_d(xr + 3 * q, phi);
        const double wq = wr[q] * taub[q];
#pragma unroll
        for (int j = 0; j < 3; ++j) t[j] = wq * (A.g[j] - gq[j]);
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int j = 0; j < 3; ++j) s[3 * a + j] = fma(phi[a], t[j], s[3 * a + j]);
    }
    // lanes with bit 4, 3, 2 set keep the upper half of the corners, the others the lower half
#pragma unroll
    for (int h = 12, o = 16; h >= 3; h /= 2, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int j = 0; j < 12; ++j)
            if (j < h) {
                const double keep = up ? s[h + j] : s[j], give = up ? s[j] : s[h + j];
                s[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
    }
    double r = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        double x = s[j];
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        x += __shfl_xor_sync(0xffffffffu, x, 2);
        if (k == j) r = x;
    }
    const double* P = pen + 36 * i;   // as in nitsche_penalty
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const int lo = c < b ? c : b, hi = c < b ? b : c;
        r = fma(P[lo * 8 - lo * (lo - 1) / 2 + hi - lo], __shfl_sync(0xffffffffu, dc, 4 * b + k), r);
    }
    r *= cbmu;
    if (A.ss) {
        if (k < 3) A.ss[32 * pslot[i] + lane] += r;
    } else {
        double rr[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int j = 0; j < 3; ++j) rr[j] = __shfl_sync(0xffffffffu, r, (lane & ~3) + j);
        if (k == 0) scatter(A, id, rr);
    }
}

// ------------------------------------------------------------------------------------------
// strong rows
// ------------------------------------------------------------------------------------------
__global__ void strong_rows(Args A, const uint8_t* __restrict__ flag, const uint8_t* __restrict__ umask,
                            const double* __restrict__ uval, double ux, double uy, double uz, int jv) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= A.n_nodes) return;
    if (A.skip && *A.skip) return;   // a captured solver step after its cycle ended
    const uint8_t f = flag[n];
    uint8_t mask;
    double gv[4];
    if (umask) {
        mask = umask[n];
        for (int k = 0; k < 4; ++k) gv[k] = uval[4 * n + k];
    } else {
        mask = f & 15;
        gv[0] = ux; gv[1] = uy; gv[2] = uz; gv[3] = 0.0;
    }
    if (f & 16) {
        for (int k = 0; k < 4; ++k)
            if (!((mask >> k) & 1)) { mask |= (uint8_t)(1 << k); gv[k] = k < 3 ? A.g[k] : 0.0; }
    }
    if (!mask) return;
    const double* src = jv ? A.V : A.U;
    for (int k = 0; k < 4; ++k)
        if ((mask >> k) & 1) A.out[4 * n + k] = jv ? src[4 * n + k] : src[4 * n + k] - gv[k];
}

// float-float accumulation on the FP32 pipe (Knuth's TwoSum): hi + lo carries the sum of floats to
// about 48 bits, in a fixed order
__device__ __forceinline__ void ff_add(float& hi, float& lo, float x) {
    const float s = __fadd_rn(hi, x);
    const float bp = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
    hi = s;
    lo = __fadd_rn(lo, e);
}

// Deterministic o2n (Algorithm 2): a thread per node sums the slot rows of its incidence list in list order
// (a hanging corner's rows times 1/2 or 1/4 for each parent; float-float in mixed precision), then the
// node's strong rows take U - g (R) or v (J v) as in strong_rows.  Bound by the latency of two dependent
// loads per entry (code, then a 16-byte row), so what counts is loads in flight: the rows of 8 entries go
// by cp.async to the thread's own places in shared memory, which takes no registers (1,280 nodes in flight
// per SM instead of 768).  Lists are padded to whole batches of 8 codes, two 16-byte loads.  Most nodes
// have one batch; the others (parents of hanging nodes, nodes at a surface: up to a hundred entries)
// would hold up their warp, so they are taken apart, longest first, in blocks of their own that start
// first; where they are few, by four lanes per node with 32 entries in flight.  Writes every row of out: no zeroing
// before the call.  2.0 M elements, mixed: 137 -> 103 us (376 MB, 3.7 TB/s); 12
// spheres: 81 -> 50 us.
constexpr int kGatherThreads = 128;
constexpr int kQuadLists = 256;   // per SM

// component k of node n after its strong rows
struct StrongRows {
    const uint8_t *flag, *umask;
    const double* uval;
    double ux, uy, uz;
    int jv;
    __device__ __forceinline__ uint8_t mask(int64_t n) const {
        const uint8_t f = flag[n];
        return (f & 16) ? 15 : umask ? umask[n] : (uint8_t)(f & 15);
    }
    __device__ __forceinline__ double row(const Args& A, int64_t n, int k) const {
        if (jv) return A.V[4 * n + k];
        const uint8_t m = umask ? umask[n] : (uint8_t)(flag[n] & 15);
        double g;
        if (!((m >> k) & 1)) g = k < 3 ? A.g[k] : 0.0;   // only because no active element reaches the node
        else if (umask) g = uval[4 * n + k];
        else g = k == 0 ? ux : k == 1 ? uy : k == 2 ? uz : 0.0;
        return A.U[4 * n + k] - g;
    }
};

template <class T, bool QUADS>
__global__ void __launch_bounds__(kGatherThreads, sizeof(T) == 4 ? 10 : 6) node_gather(
    Args A, const uint32_t* __restrict__ head, const int32_t* __restrict__ heavy, const int64_t* __restrict__ hptr,
    const uint32_t* __restrict__ inc, int64_t n_heavy, unsigned heavy_blocks, int64_t nv, StrongRows S) {
    static_assert(kIncHead == 8, "batches of two 16-byte loads");
    constexpr int C = sizeof(T) / 4;   // 16-byte chunks of a row
    __shared__ __align__(16) uint4 s_row[8][C][kGatherThreads];
    __shared__ uint32_t s_code[QUADS ? 8 : 1][kGatherThreads];
    if (A.skip && *A.skip) return;   // a captured solver step after its cycle ended
    if (QUADS && blockIdx.x < heavy_blocks) {
        // four lanes per node: each fetches the rows of 8 of the next 32 entries, then sums one component of
        // all 32 in order
        const int64_t h = ((int64_t)blockIdx.x * kGatherThreads + threadIdx.x) >> 2;
        const int k = threadIdx.x & 3, quad = threadIdx.x & ~3;
        const bool live = h < n_heavy;
        const int64_t q1 = live ? hptr[h + 1] : 0;
        int64_t q = live ? hptr[h] : 0;
        double acc = 0.0;
        float hi = 0.f, lo = 0.f;
        for (; __any_sync(0xffffffffu, q < q1); q += 32) {
            const int64_t mine = q + 8 * k;
            uint4 c[2] = {{kIncNone, kIncNone, kIncNone, kIncNone}, {kIncNone, kIncNone, kIncNone, kIncNone}};
            if (mine < q1) {
                c[0] = __ldg(reinterpret_cast<const uint4*>(inc + mine));
                c[1] = __ldg(reinterpret_cast<const uint4*>(inc + mine) + 1);
            }
            const uint32_t e[8] = {c[0].x, c[0].y, c[0].z, c[0].w, c[1].x, c[1].y, c[1].z, c[1].w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int64_t sl = (int64_t)(e[i] >> 5);
                s_code[QUADS ? i : 0][threadIdx.x] = e[i];
                if (sl < nv) {   // (a padding code's slot is past every volume slot)
                    const char* r = (const char*)A.sv + (32 * sl + 4 * (e[i] & 7)) * sizeof(T);
#pragma unroll
                    for (int b = 0; b < C; ++b) cp16(&s_row[i][b][threadIdx.x], r + 16 * b);
                }
            }
            cp_commit();
            cp_wait<0>();
            __syncwarp();
            for (int f = 0; f < 4 && q + 8 * f < q1; ++f)
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t code = s_code[QUADS ? i : 0][quad + f];
                    if (code == kIncNone) continue;
                    const int wc = (int)((code >> 3) & 3);
                    const int64_t sl = (int64_t)(code >> 5);
                    if (sl < nv) {
                        const T w = wc == 0 ? T(1) : (wc == 1 ? T(0.5) : T(0.25));
                        const T v = reinterpret_cast<const T*>(&s_row[i][k * sizeof(T) / 16][quad + f])[k & (16 / sizeof(T) - 1)];
                        if constexpr (sizeof(T) == 4) ff_add(hi, lo, w * v);
                        else acc += w * v;
                    } else {   // a float64 surface slot
                        const double w = wc == 0 ? 1.0 : (wc == 1 ? 0.5 : 0.25);
                        acc += w * A.ss[32 * (sl - nv) + 4 * (code & 7) + k];
                    }
                }
            __syncwarp();   // the rows and codes are replaced
        }
        if (!live) return;
        const int64_t n = heavy[h];
        if constexpr (sizeof(T) == 4) acc += f2d(hi) + f2d(lo);
        A.out[4 * n + k] = (S.mask(n) >> k) & 1 ? S.row(A, n, k) : acc;
        return;
    }
    int64_t n;
    const uint4* code;
    int batches = 1;
    if (blockIdx.x < heavy_blocks) {
        const int64_t h = (int64_t)blockIdx.x * kGatherThreads + threadIdx.x;
        if (h >= n_heavy) return;
        n = heavy[h];
        const int64_t q0 = hptr[h];
        batches = (int)((hptr[h + 1] - q0) >> 3);
        code = reinterpret_cast<const uint4*>(inc + q0);
    } else {
        n = (int64_t)(blockIdx.x - heavy_blocks) * kGatherThreads + threadIdx.x;
        if (n >= A.n_nodes) return;
        code = reinterpret_cast<const uint4*>(head + kIncHead * n);
    }
    uint4 h0 = __ldg(code), h1 = __ldg(code + 1);
    if (h0.x == kIncHeavy) return;
    const uint8_t mask = S.mask(n);
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
    bool surf = false;
    for (;;) {
        const uint32_t e[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int64_t sl = (int64_t)(e[i] >> 5);
            if (sl < nv) {   // (a padding code's slot is past every volume slot)
                const char* r = (const char*)A.sv + (32 * sl + 4 * (e[i] & 7)) * sizeof(T);
#pragma unroll
                for (int c = 0; c < C; ++c) cp16(&s_row[i][c][threadIdx.x], r + 16 * c);
            }
        }
        cp_commit();
        if (--batches > 0) {   // the next codes arrive beside the rows
            code += 2;
            h0 = __ldg(code);
            h1 = __ldg(code + 1);
        }
        cp_wait<0>();   // this thread's own copies
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (e[i] == kIncNone) continue;
            const int c = (int)(e[i] & 7), wc = (int)((e[i] >> 3) & 3);
            const int64_t sl = (int64_t)(e[i] >> 5);
            if (sl < nv) {
                const T w = wc == 0 ? T(1) : (wc == 1 ? T(0.5) : T(0.25));
                if constexpr (sizeof(T) == 4) {
                    const float4 v = *reinterpret_cast<const float4*>(&s_row[i][0][threadIdx.x]);
                    ff_add(hi[0], lo[0], w * v.x);
                    ff_add(hi[1], lo[1], w * v.y);
                    ff_add(hi[2], lo[2], w * v.z);
                    ff_add(hi[3], lo[3], w * v.w);
                } else {
                    const double2 x = *reinterpret_cast<const double2*>(&s_row[i][0][threadIdx.x]),
                                  y = *reinterpret_cast<const double2*>(&s_row[i][C - 1][threadIdx.x]);
                    acc[0] += w * x.x; acc[1] += w * x.y; acc[2] += w * y.x; acc[3] += w * y.y;
                }
            } else {   // a float64 surface slot
                const double* d = A.ss + 32 * (sl - nv) + 4 * c;
                const double2 x = reinterpret_cast<const double2*>(d)[0], y = reinterpret_cast<const double2*>(d)[1];
                const double w = wc == 0 ? 1.0 : (wc == 1 ? 0.5 : 0.25);
                acc[0] += w * x.x; acc[1] += w * x.y; acc[2] += w * y.x; acc[3] += w * y.y;
                surf = true;
            }
        }
        if (batches <= 0) break;
    }
    if constexpr (sizeof(T) == 4)
        for (int k = 0; k < 4; ++k) {
            const double s = f2d(hi[k]) + f2d(lo[k]);
            acc[k] = surf ? acc[k] + s : s;
        }
    if (mask)
        for (int k = 0; k < 4; ++k)
            if ((mask >> k) & 1) acc[k] = S.row(A, n, k);
    double2* o = reinterpret_cast<double2*>(A.out + 4 * n);
    o[0] = make_double2(acc[0], acc[1]);
    o[1] = make_double2(acc[2], acc[3]);
}

// optional event pair around a launch (profiling); never for calls on a caller's workspace
// (imga_jvp_noalloc), which create no events and leave the mesh untouched
struct Timed {
    Mesh* m;
    int k, nk;
    cudaStream_t s;
    cudaEvent_t a = nullptr, b = nullptr;
    Timed(const Mesh& mesh, int kind, cudaStream_t st, int launches = 1, bool enable = true)
        : m(const_cast<Mesh*>(&mesh)), k(kind), nk(launches), s(st) {
        if (!enable || !m->profiling) return;
        cudaEventCreate(&a);
        cudaEventCreate(&b);
        cudaEventRecord(a, s);
    }
    ~Timed() {
        if (!a) return;
        cudaEventRecord(b, s);
        m->prof_ev[k].push_back({(void*)a, (void*)b, nk});
    }
};

bool cut_is_split(const Mesh& m) { return (int64_t)m.cut_list.size() <= (int64_t)kSplitCut * m.n_sm; }   // float32

template <class T, bool JV>
void launch_cut(const Mesh& m, const Args& A, cudaStream_t s, int wpb, int lpt, bool generic = false) {
    const int64_t nc = (int64_t)m.cut_list.size();
    const int32_t* order = lpt ? m.d.cut_order : nullptr;
    if constexpr (sizeof(T) == 8) {
        if (generic) vms_cut_split<T, JV><<<(unsigned)nc, 128, 0, s>>>(A, m.d.cut_list, m.d.cut_off, m.d.cut_pts, order);
        else if (wpb == 2) vms_cut64<JV, 2><<<(unsigned)nc, 64, 0, s>>>(A, m.d.cut_list, m.d.cut_off, m.d.cut_pts, order);
        else vms_cut64<JV, 4><<<(unsigned)nc, 128, 0, s>>>(A, m.d.cut_list, m.d.cut_off, m.d.cut_pts, order);
    } else {
        const void* pts = m.d.cut_pts_f;
        if (cut_is_split(m)) {
            vms_cut_split<T, JV><<<(unsigned)nc, 128, 0, s>>>(A, m.d.cut_list, m.d.cut_off, pts, order);
            return;
        }
        switch (wpb) {
            case 2: vms_cut<JV, 2><<<(unsigned)((nc + 1) / 2), 64, 0, s>>>(A, m.d.cut_list, m.d.cut_off, pts, order, nc); break;
            case 8: vms_cut<JV, 8><<<(unsigned)((nc + 7) / 8), 256, 0, s>>>(A, m.d.cut_list, m.d.cut_off, pts, order, nc); break;
            default: vms_cut<JV, 4><<<(unsigned)((nc + 3) / 4), 128, 0, s>>>(A, m.d.cut_list, m.d.cut_off, pts, order, nc);
        }
    }
}

template <class T, bool JV, int MINB = (sizeof(T) == 4 ? 4 : 2), bool GEN = false>
int interior_blocks_per_sm();
template <class T, bool JV>
void launch_interior(const Mesh& m, const Args& A, cudaStream_t s, int bps, bool generic = false);

// Autotuner of the Intercepted-element bucket: with the node data of this call prepared, time every
// (warps per block, element order) candidate on the call's own inputs (3 launches each after one
// untimed) and keep the fastest; then the Out-element bucket: the persistent interior kernel with
// 1 .. 4 resident blocks per SM, and 5 with the smaller register allocation (float).  Writes into the output vector, which the call then recomputes.
template <class T, bool JV>
int autotune_cut(Mesh& m, Args A, cudaStream_t s) {
    const int64_t nc = (int64_t)m.cut_list.size();
    Mesh::CutTune& ct = m.cut_tune[sizeof(T) == 4][JV];
    m.tune_pending[sizeof(T) == 4][JV] = false;
    const int64_t next = m.n_nodes() + m.n_hang();
    T* ndv = node_workspace<T>(m, nullptr);
    A.ndv = ndv;
    A.ndt = ndv + 8 * next;
    A.ndf = A.F ? ndv + 16 * next : nullptr;
    launch_node_prep<T, JV>(A, ndv, (T*)A.ndt, (T*)A.ndf, s);
    const int wpbs[3] = {2, 4, 8};
    const int nw = sizeof(T) == 4 ? 3 : 2;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    // (vms_cut_split has one shape, four warps: the others are not measured)
    const bool split = sizeof(T) == 4 && cut_is_split(m);
    for (int wi = split ? 1 : 0; wi < (split ? 2 : nw) && nc > 0; ++wi)
        for (int lpt = 0; lpt < 2; ++lpt) {
            launch_cut<T, JV>(m, A, s, wpbs[wi], lpt);
            cudaEventRecord(e0, s);
            for (int r = 0; r < 3; ++r) launch_cut<T, JV>(m, A, s, wpbs[wi], lpt);
            cudaEventRecord(e1, s);
            cudaEventSynchronize(e1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            ms /= 3.f;
            m.cut_tune_ms[sizeof(T) == 4][JV][2 * wi + lpt] = ms;
            if (ms < best) { best = ms; ct = {wpbs[wi], lpt, true}; }
        }
    // the Out-element bucket: the persistent interior kernel with 1 .. (occupancy limit) blocks per SM
    const int64_t no = (int64_t)m.out_list.size();
    constexpr int EPB = Epb<T>::value;
    int maxb = std::min(4, interior_blocks_per_sm<T, JV>());
    if constexpr (sizeof(T) == 4)
        if (maxb == 4 && interior_blocks_per_sm<T, JV, 5>() >= 5) maxb = 5;
    float best_out = 1e30f;
    for (int b = 1; b <= maxb && no > 0; ++b) {
        auto run = [&]() { launch_interior<T, JV>(m, A, s, b); };
        run();
        cudaEventRecord(e0, s);
        for (int r = 0; r < 3; ++r) run();
        cudaEventRecord(e1, s);
        cudaEventSynchronize(e1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        ms /= 3.f;
        m.out_tune_ms[sizeof(T) == 4][JV][b - 1] = ms;
        if (ms < best_out) { best_out = ms; m.out_bps[sizeof(T) == 4][JV] = b; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

// Resident CTAs of the persistent interior kernel per SM (queried once; also sets its dynamic smem opt-in).
template <class T, bool JV, int MINB, bool GEN>
int interior_blocks_per_sm() {
    static int bps = 0;
    if (bps == 0) {
        const size_t smem = IntShape<T>::smem;
        int b = 0;
        cudaFuncSetAttribute(vms_interior<T, JV, MINB, GEN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, vms_interior<T, JV, MINB, GEN>, 8 * Epb<T>::value, smem);
        bps = b < 1 ? 1 : b;
    }
    return bps;
}

// The persistent interior kernel at bps resident blocks per SM: the 5-block register allocation for
// bps = 5 (float only), else the default one.
template <class T, bool JV>
void launch_interior(const Mesh& m, const Args& A, cudaStream_t s, int bps, bool generic) {
    const int64_t no = (int64_t)m.out_list.size();
    constexpr int EPB = Epb<T>::value;
    const int64_t grid = std::min<int64_t>((no + EPB - 1) / EPB, (int64_t)bps * m.n_sm);
    if constexpr (sizeof(T) == 4) {
        if (bps >= 5) {
            vms_interior<T, JV, 5><<<(unsigned)grid, 8 * EPB, IntShape<T>::smem, s>>>(A, m.d.out_conn, m.d.out_lev, m.d.out_prob, no);
            return;
        }
    }
    if constexpr (sizeof(T) == 8) {
        if (generic) {
            vms_interior<T, JV, 2, true><<<(unsigned)grid, 8 * EPB, IntShape<T>::smem, s>>>(A, m.d.out_conn, m.d.out_lev, m.d.out_prob, no);
            return;
        }
    }
    vms_interior<T, JV><<<(unsigned)grid, 8 * EPB, IntShape<T>::smem, s>>>(A, m.d.out_conn, m.d.out_lev, m.d.out_prob, no);
}

// Resident CTAs of the fused kernel per SM (queried once; also sets its dynamic smem opt-in).
template <class T, bool JV, bool GEN = false>
int fused_blocks_per_sm() {
    static int bps = 0;
    if (bps == 0) {
        const size_t smem = FusedShape<T>::smem;
        int b = 0;
        cudaFuncSetAttribute(vms_fused<T, JV, GEN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, vms_fused<T, JV, GEN>, 32 * kFusedWarps, smem);
        bps = b < 1 ? 1 : b;
    }
    return bps;
}

template <class T, bool JV>
void launch_penalty(const Mesh& m, const Args& A, cudaStream_t s, bool timed) {
    const int64_t np = (int64_t)m.pen_elem.size();
    if (np <= 0) return;
    Timed t(m, 2, s, 1, timed);
    if (!JV && A.gpts)
        nitsche_penalty_points<<<(unsigned)((np + 3) / 4), 128, 0, s>>>(A, m.d.pen_elem, m.d.pen_q, m.d.pen_slot, m.d.pen,
                                                                        m.d.sq_x, m.d.sq_w, m.d.sq_taub, np);
    else
        nitsche_penalty<JV><<<(unsigned)((8 * np + 127) / 128), 128, 0, s>>>(A, m.d.pen_elem, m.d.pen_slot, m.d.pen, np);
}

// the surface buckets: thread-per-point and warp-per-element Nitsche kernels, then the float64
// penalty (same stream: the slots hold their rows first)
template <class T, bool JV>
void launch_surface(const Mesh& m, const Args& A, cudaStream_t ss, bool timed) {
    const int64_t nsp = m.n_sq_sparse, nse = m.n_sq_elem;
    if (nsp > 0) {
        Timed t(m, 2, ss, 1, timed);
        nitsche<T, JV><<<(unsigned)((nsp + 127) / 128), 128, 0, ss>>>(A, m.d.sq_elem, m.d.sq_x, m.d.sq_n, m.d.sq_w,
                                                                      m.d.sq_taub, nsp);
    }
    if (nse > 0) {
        Timed t(m, 2, ss, 1, timed);
        nitsche_el<T, JV><<<(unsigned)((nse + WPB - 1) / WPB), 32 * WPB, 0, ss>>>(A, m.d.sq_list, m.d.sq_off, m.d.sq_x,
                                                                                m.d.sq_n, m.d.sq_w, m.d.sq_taub, nse);
    }
    launch_penalty<T, JV>(m, A, ss, timed);
}

// the Out and Intercepted buckets in one persistent launch (vms_fused); the surface kernels beside
// it on the side stream ss (forked and joined with the events ev), or after it on s
template <class T, bool JV>
void launch_fused(const Mesh& m, const Args& A, cudaStream_t s, cudaStream_t ss, cudaEvent_t* ev, bool timed, bool generic) {
    const bool fork = ev && ss && ss != s;
    if (fork) {   // the surface kernels first: their blocks take their SMs, the persistent queue fills the rest
        cudaEventRecord(ev[0], s);
        cudaStreamWaitEvent(ss, ev[0], 0);
        launch_surface<T, JV>(m, A, ss, timed);
    }
    FusedQueue Q;
    Q.items = m.d.fq_items;
    Q.n_items = m.fq_n;
    Q.cnt = m.d.fq_cnt;
    Q.oconn = m.d.out_conn;
    Q.olev = m.d.out_lev;
    Q.oprob = m.d.out_prob;
    Q.n_out = (int64_t)m.out_list.size();
    Q.cut_list = m.d.cut_list;
    Q.cut_off = m.d.cut_off;
    Q.cut_pts = std::is_same<T, float>::value ? (const void*)m.d.cut_pts_f : (const void*)m.d.cut_pts;
    Q.heavy_warps = m.fused_heavy_warps;
    if (Q.n_items + Q.n_out > 0) {
        Timed t(m, 5, s, 1, timed);
        const int64_t work = Q.n_items + (Q.n_out + 3) / 4;   // warp items
        const int64_t blocks = (work + kFusedWarps - 1) / kFusedWarps;
        auto run = [&](auto kernel, int bps) {
            kernel<<<(unsigned)std::min<int64_t>(blocks, (int64_t)bps * m.n_sm), 32 * kFusedWarps, FusedShape<T>::smem, s>>>(A, Q);
        };
        if constexpr (sizeof(T) == 8) {
            if (generic) run(vms_fused<T, JV, true>, fused_blocks_per_sm<T, JV, true>());
            else run(vms_fused<T, JV>, fused_blocks_per_sm<T, JV>());
        } else {
            run(vms_fused<T, JV>, fused_blocks_per_sm<T, JV>());
        }
    }
    if (fork) {
        cudaEventRecord(ev[2], ss);
        cudaStreamWaitEvent(s, ev[2], 0);
    } else {
        launch_surface<T, JV>(m, A, s, timed);
    }
}

template <class T, bool JV>
void launch_all(const Mesh& m, Args A, cudaStream_t s, void* ws = nullptr, cudaStream_t s_cut = nullptr,
                cudaStream_t s_sur = nullptr, cudaEvent_t* ev = nullptr, bool generic = false) {
    const int64_t next = m.n_nodes() + m.n_hang();
    T* ndv = node_workspace<T>(m, ws);
    T* ndt = ndv + 8 * next;
    T* ndf = A.F ? ndt + 8 * next : nullptr;
    A.ndv = ndv;
    A.ndt = ndt;
    A.ndf = ndf;
    if (next > 0) {
        Timed t(m, 4, s, (A.n_nodes > 0) + (A.n_hang > 0), !ws);
        launch_node_prep<T, JV>(A, ndv, ndt, ndf, s);
    }
    if (m.fused && m.d.fq_cnt) {
        launch_fused<T, JV>(m, A, s, s_sur, ev, !ws, generic);
        return;
    }
    // fork: the Intercepted-element and surface kernels run beside the Out-element kernel
    const cudaStream_t sc = s_cut ? s_cut : s, ss = s_sur ? s_sur : s;
    if (ev) {
        cudaEventRecord(ev[0], s);
        cudaStreamWaitEvent(sc, ev[0], 0);
        cudaStreamWaitEvent(ss, ev[0], 0);
    }
    const int64_t no = (int64_t)m.out_list.size(), nc = (int64_t)m.cut_list.size();
    constexpr int EPB = Epb<T>::value;
    if (no > 0) {
        Timed t(m, 0, s, 1, !ws);
        const int tuned = m.out_bps[sizeof(T) == 4][JV];
        launch_interior<T, JV>(m, A, s, tuned > 0 ? tuned : interior_blocks_per_sm<T, JV>(), generic);
    }
    if (nc > 0) {
        Timed t(m, 1, sc, 1, !ws);
        const Mesh::CutTune& ct = m.cut_tune[sizeof(T) == 4][JV];
        launch_cut<T, JV>(m, A, sc, ct.wpb, ct.lpt || !ct.tuned, generic);
    }
    launch_surface<T, JV>(m, A, ss, !ws);
    if (ev) {   // join
        cudaEventRecord(ev[1], sc);
        cudaEventRecord(ev[2], ss);
        cudaStreamWaitEvent(s, ev[1], 0);
        cudaStreamWaitEvent(s, ev[2], 0);
    }
}

// strong rows; with the deterministic scatter, the node sums (which write every row) and the strong rows
void launch_strong_rows(const Mesh& m, const Args& A, const imga_physics& ph, bool jv, cudaStream_t s,
                        bool timed = true, int precision = 0) {
    const int64_t nn = m.n_nodes();
    Timed t(m, 3, s, 1, timed);
    if (nn > 0 && A.sv) {
        const uint8_t* um = m.user_bc ? m.d.bcmask_user : nullptr;
        const double* uv = m.user_bc ? m.d.bcval_user : nullptr;
        const StrongRows S = {m.d.bcflag, um, uv, ph.u_inf[0], ph.u_inf[1], ph.u_inf[2], jv ? 1 : 0};
        // long lists by four lanes per node where that still leaves the chip idle, by a thread per node else
        // (4 k lists: 17 us against 26; 350 k lists: 58 against 50)
        const bool quads = m.n_heavy <= (int64_t)kQuadLists * m.n_sm;
        const unsigned hb = (unsigned)(((quads ? 4 : 1) * m.n_heavy + kGatherThreads - 1) / kGatherThreads),
                       grid = hb + (unsigned)((nn + kGatherThreads - 1) / kGatherThreads);
        auto run = [&](auto kernel) {
            kernel<<<grid, kGatherThreads, 0, s>>>(A, m.d.inc_head, m.d.inc_heavy, m.d.inc_ptr, m.d.inc, m.n_heavy, hb, m.n_vslots, S);
        };
        if (precision == 0) { if (quads) run(node_gather<double, true>); else run(node_gather<double, false>); }
        else { if (quads) run(node_gather<float, true>); else run(node_gather<float, false>); }
        return;
    }
    if (nn > 0)
        strong_rows<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(A, m.d.bcflag, m.user_bc ? m.d.bcmask_user : nullptr,
                                                                m.user_bc ? m.d.bcval_user : nullptr, ph.u_inf[0],
                                                                ph.u_inf[1], ph.u_inf[2], jv ? 1 : 0);
}

}  // namespace

// The work queue of the fused launch: the Intercepted elements by decreasing point count (the cost
// of an element on a warp is its rounds of 32 sub-cell points, Eq. Wpart's volume term), claimed
// first; the Out elements follow in Morton order, claimed in chunks.
int fused_prepare(Mesh& m, std::string& err) {
    const int64_t nc = (int64_t)m.cut_list.size();
    std::vector<uint32_t> items((size_t)nc);
    for (int64_t i = 0; i < nc; ++i) items[i] = (uint32_t)i;
    std::stable_sort(items.begin(), items.end(), [&](uint32_t a, uint32_t b) {
        return m.cut_off[a + 1] - m.cut_off[a] > m.cut_off[b + 1] - m.cut_off[b];
    });
    if (m.d.fq_items) { cudaFree(m.d.fq_items); m.d.fq_items = nullptr; }
    if (m.d.fq_cnt) { cudaFree(m.d.fq_cnt); m.d.fq_cnt = nullptr; }
    if (cudaMalloc((void**)&m.d.fq_items, std::max<size_t>(1, items.size()) * sizeof(uint32_t)) != cudaSuccess ||
        cudaMalloc((void**)&m.d.fq_cnt, 3 * sizeof(unsigned long long)) != cudaSuccess ||
        (!items.empty() && cudaMemcpy(m.d.fq_items, items.data(), items.size() * sizeof(uint32_t), cudaMemcpyHostToDevice) != cudaSuccess) ||
        cudaMemset(m.d.fq_cnt, 0, 3 * sizeof(unsigned long long)) != cudaSuccess) {
        err = "fused queue upload";
        return 1;
    }
    m.fq_n = nc;
    m.fq_counts[0] = nc;
    m.fq_counts[1] = m.n_sq_elem;
    m.fq_counts[2] = m.n_sq_sparse;
    fused_blocks_per_sm<double, true>();
    fused_blocks_per_sm<double, false>();
    fused_blocks_per_sm<double, true, true>();
    fused_blocks_per_sm<double, false, true>();
    fused_blocks_per_sm<float, true>();
    fused_blocks_per_sm<float, false>();
    return 0;
}

void graphs_free(Mesh& m) {
    for (auto& g : m.graphs) cudaGraphExecDestroy((cudaGraphExec_t)g.second);
    m.graphs.clear();
    for (int k = 0; k < 3; ++k) if (m.side[k]) { cudaStreamDestroy((cudaStream_t)m.side[k]); m.side[k] = nullptr; }
    for (int k = 0; k < 5; ++k) if (m.fork_ev[k]) { cudaEventDestroy((cudaEvent_t)m.fork_ev[k]); m.fork_ev[k] = nullptr; }
}

// the mesh's side streams and fork / join events (created on first use)
int side_streams(Mesh& mm) {
    if (mm.side[0]) return 0;
    for (int k = 0; k < 3; ++k)
        if (cudaStreamCreateWithFlags((cudaStream_t*)&mm.side[k], cudaStreamNonBlocking) != cudaSuccess) return 1;
    for (int k = 0; k < 5; ++k)
        if (cudaEventCreateWithFlags((cudaEvent_t*)&mm.fork_ev[k], cudaEventDisableTiming) != cudaSuccess) return 1;
    return 0;
}

static int vms_apply_ws(const Mesh& m, const double* u, const double* up, const double* up2, const double* f,
                        const imga_physics& ph, int precision, const double* v, double* out, void* stream, void* ws,
                        bool generic) {
    cudaStream_t s = (cudaStream_t)stream;
    Args A = make_args(m, u, up, up2, f, ph, v, out);
    const bool jv = v != nullptr;
    if (generic) {   // (launch attributes, once)
        interior_blocks_per_sm<double, true, 2, true>();
        interior_blocks_per_sm<double, false, 2, true>();
    }
    if (m.tune_pending[precision != 0][jv] && !ws) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        cudaStreamIsCapturing(s, &cs);
        if (cs == cudaStreamCaptureStatusNone) {
            Mesh& mm = const_cast<Mesh&>(m);
            const int rc = precision == 0 ? (jv ? autotune_cut<double, true>(mm, A, s) : autotune_cut<double, false>(mm, A, s))
                                          : (jv ? autotune_cut<float, true>(mm, A, s) : autotune_cut<float, false>(mm, A, s));
            if (rc) return 1;
            graphs_free(mm);   // captured launches carry the old tile shapes
        }
    }
    if (m.use_graphs && !ws && !m.profiling) {
        // Replay (or capture once) the whole call as a CUDA graph with parallel branches.  Capture runs on
        // a private stream (the legacy default stream cannot be captured); the graph is launched on a
        // private stream too, ordered after the caller's stream by events and joined back into it.
        Mesh& mm = const_cast<Mesh&>(m);
        GraphKey key;
        std::memset(&key, 0, sizeof(key));
        key.u = u; key.up = up; key.up2 = up2; key.f = f; key.v = v; key.out = out;
        key.precision = precision | (generic ? 2 : 0);
        key.ph = ph;
        key.user_bc = m.user_bc;
        if (side_streams(mm)) return 1;
        cudaStream_t s1 = (cudaStream_t)mm.side[0], s2 = (cudaStream_t)mm.side[1], cs = (cudaStream_t)mm.side[2];
        cudaEvent_t* ev = (cudaEvent_t*)mm.fork_ev;
        cudaGraphExec_t exec = nullptr;
        for (auto& g : mm.graphs)
            if (std::memcmp(&g.first, &key, sizeof(key)) == 0) { exec = (cudaGraphExec_t)g.second; break; }
        if (!exec) {
            vms_prepare();
            cudaGraph_t graph = nullptr;
            if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return 1;
            if (!A.sv) cudaMemsetAsync(out, 0, (size_t)m.n_nodes() * 4 * sizeof(double), cs);
            cudaStream_t b1 = m.concurrent ? s1 : cs, b2 = m.concurrent ? s2 : cs;
            cudaEvent_t* bev = m.concurrent ? ev : nullptr;
            if (precision == 0) {
                if (jv) launch_all<double, true>(m, A, cs, nullptr, b1, b2, bev, generic); else launch_all<double, false>(m, A, cs, nullptr, b1, b2, bev, generic);
            } else {
                if (jv) launch_all<float, true>(m, A, cs, nullptr, b1, b2, bev); else launch_all<float, false>(m, A, cs, nullptr, b1, b2, bev);
            }
            launch_strong_rows(m, A, ph, jv, cs, true, precision);
            const cudaError_t ec = cudaStreamEndCapture(cs, &graph);
            if (ec != cudaSuccess || !graph) return 1;
            const cudaError_t rc = cudaGraphInstantiate(&exec, graph, 0);
            cudaGraphDestroy(graph);
            if (rc != cudaSuccess) return 1;
            if (mm.graphs.size() >= 32) {   // bounded cache: drop the oldest
                cudaGraphExecDestroy((cudaGraphExec_t)mm.graphs.front().second);
                mm.graphs.erase(mm.graphs.begin());
            }
            mm.graphs.push_back({key, (void*)exec});
        }
        if (cudaEventRecord(ev[3], s) != cudaSuccess || cudaStreamWaitEvent(cs, ev[3], 0) != cudaSuccess) return 1;
        if (cudaGraphLaunch(exec, cs) != cudaSuccess) return 1;
        if (cudaEventRecord(ev[4], cs) != cudaSuccess || cudaStreamWaitEvent(s, ev[4], 0) != cudaSuccess) return 1;
        return 0;
    }
    if (!A.sv && cudaMemsetAsync(out, 0, (size_t)m.n_nodes() * 4 * sizeof(double), s) != cudaSuccess) return 1;
    // the Intercepted-element and surface kernels on the mesh's side streams, beside the Out-element
    // kernel, as in the captured graph (not for calls on a caller's workspace, which create nothing)
    cudaStream_t s1 = nullptr, s2 = nullptr;
    cudaEvent_t* ev = nullptr;
    if (!ws && m.concurrent) {
        Mesh& mm = const_cast<Mesh&>(m);
        if (side_streams(mm)) return 1;
        s1 = (cudaStream_t)mm.side[0];
        s2 = (cudaStream_t)mm.side[1];
        ev = (cudaEvent_t*)mm.fork_ev;
    }
    if (precision == 0) {
        if (jv) launch_all<double, true>(m, A, s, ws, s1, s2, ev, generic); else launch_all<double, false>(m, A, s, ws, s1, s2, ev, generic);
    } else {
        if (jv) launch_all<float, true>(m, A, s, ws, s1, s2, ev); else launch_all<float, false>(m, A, s, ws, s1, s2, ev);
    }
    launch_strong_rows(m, A, ph, jv, s, !ws, precision);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

// ------------------------------------------------------------------------------------------
// Force of the fluid on the body: the surface terms of Eq. (weakbc) tested with w = e_i, i.e. summed
// over every node's momentum rows (partition of unity), in float64.  Per surface point
//   w_q [ -(sigma(u_s, p) n)_i - [u.n < 0] rho (u.n) (u - g)_i + tau_B (u - g)_i ],
// n the fluid-outward normal: the force that keeps the discrete momentum balance of weak Dirichlet
// conditions.  Each block sums its points in a fixed order, then one block sums the partials in
// block order (same bits on every call).
// ------------------------------------------------------------------------------------------
constexpr int kForceBlocks = 256;

__global__ void __launch_bounds__(256) surface_force_partial(Args A, const int32_t* __restrict__ el,
                                                             const double* __restrict__ xr, const double* __restrict__ nr,
                                                             const double* __restrict__ wr, const double* __restrict__ taub,
                                                             int64_t n, double* __restrict__ part) {
    double f[3] = {0.0, 0.0, 0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        NitschePoint<double, double> P;
        nitsche_fields<double, double, false>(A, el[i], i, xr + 3 * i, nr + 3 * i, P);
        const double tauB = A.Cb * P.mu * taub[i];
        for (int k = 0; k < 3; ++k) {
            double t = -P.tr[k] + tauB * P.dd[k];
            if (P.inflow) t -= P.rho * P.un * P.dd[k];
            f[k] += wr[i] * t;
        }
    }
    __shared__ double red[3][8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int k = 0; k < 3; ++k) {
        double v = f[k];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[k][wid] = v;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double v = 0.0;
        for (int j = 0; j < (int)(blockDim.x >> 5); ++j) v += red[threadIdx.x][j];
        part[3 * blockIdx.x + threadIdx.x] = v;
    }
}

__global__ void surface_force_final(int nb, const double* __restrict__ part, double* __restrict__ F) {
    if (threadIdx.x >= 3) return;
    double v = 0.0;
    for (int b = 0; b < nb; ++b) v += part[3 * b + threadIdx.x];
    F[threadIdx.x] = v;
}

// ------------------------------------------------------------------------------------------
// self-check of f2d / d2f against the hardware conversions
// ------------------------------------------------------------------------------------------
namespace {
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void conversion_check(int64_t n, uint64_t seed, unsigned long long* bad) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t r = mix64(seed + 0x9E3779B97F4A7C15ull * (uint64_t)(i + 1));
    const uint64_t r2 = mix64(r ^ 0xD1B54A32D192ED03ull);
    uint64_t bits;
    const uint64_t sign = r2 & 0x8000000000000000ull, frac = r & 0x000FFFFFFFFFFFFFull;
    switch (i & 7) {
        case 0: bits = r; break;                                                    // anything
        case 1: bits = sign | ((uint64_t)(897 + (r2 >> 8) % 254) << 52) | frac; break;   // float32 normal range
        case 2: bits = sign | ((uint64_t)(897 + (r2 >> 8) % 254) << 52) | (frac & ~0x1FFFFFFFull) | 0x10000000ull; break;  // tie
        case 3: {                                                                   // edges of the range
            const uint32_t E[6] = {0, 1, 896, 897, 1150, 1151};
            bits = sign | ((uint64_t)E[(r2 >> 8) % 6] << 52) | frac;
            break;
        }
        case 4: bits = sign | ((uint64_t)1150 << 52) | (0x000FFFFFF0000000ull | (frac & 0x0FFFFFFFull)); break;  // rounds to inf
        case 5: bits = sign | ((uint64_t)(r2 % 3 == 0 ? 2047 : (r2 % 3 == 1 ? 0 : 1)) << 52) | ((r2 >> 4) & 1 ? frac : 0); break;
        case 6: bits = sign | ((uint64_t)(897 + (r2 >> 8) % 254) << 52) | (frac | 0x000FFFFFE0000000ull); break;   // carry into the exponent
        default: bits = sign | ((uint64_t)(897 + (r2 >> 8) % 254) << 52) | (frac & ~0x1FFFFFFFull); break;        // exact in float32
    }
    const double x = __longlong_as_double((long long)bits);
    const float a = d2f(x), b = (float)x;
    bool ok = (a != a) ? (b != b) : (__float_as_uint(a) == __float_as_uint(b));
    const float y = __uint_as_float((uint32_t)(r2 >> 17));
    const double c = f2d(y), d = (double)y;
    ok = ok && ((c != c) ? (d != d) : (__double_as_longlong(c) == __double_as_longlong(d)));
    if (!ok) atomicAdd(bad, 1ull);
}
}  // namespace

int conversion_selftest(int64_t n, uint64_t seed, int64_t* mismatches, std::string& err) {
    unsigned long long* bad = nullptr;
    if (cudaMalloc((void**)&bad, sizeof(*bad)) != cudaSuccess) { err = "cudaMalloc failed"; return 1; }
    cudaMemset(bad, 0, sizeof(*bad));
    if (n > 0) conversion_check<<<(unsigned)((n + 255) / 256), 256>>>(n, seed, bad);
    unsigned long long h = 0;
    const cudaError_t rc = cudaMemcpy(&h, bad, sizeof(h), cudaMemcpyDeviceToHost);
    cudaFree(bad);
    if (rc != cudaSuccess) { err = cudaGetErrorString(rc); return 1; }
    *mismatches = (int64_t)h;
    return 0;
}

constexpr int64_t kForkOut = 65536;

// Residual / J v on `stream` without the graph path, every kernel returning at once while *skip is
// nonzero (steps of a solver loop that is itself captured in a graph).
int vms_apply_skip(const Mesh& m, const double* u, const double* up, const double* up2, const double* f,
                   const imga_physics& ph, int precision, const double* v, double* out, void* stream,
                   const int* skip, bool generic) {
    cudaStream_t s = (cudaStream_t)stream;
    Args A = make_args(m, u, up, up2, f, ph, v, out);
    A.skip = skip;
    const bool jv = v != nullptr;
    if (!A.sv && cudaMemsetAsync(out, 0, (size_t)m.n_nodes() * 4 * sizeof(double), s) != cudaSuccess) return 1;
    // a small mesh's Out kernel is a few microseconds, so its latency-bound neighbours run beside it here
    // too; from kForkOut Out elements on they gain less than the fork and join cost the captured step
    // (2.0 M elements: 1.96 s a Newton step in one stream, 2.00 s forked; 7.3 k elements: a Newton
    // solve 3 % faster forked)
    cudaStream_t s1 = nullptr, s2 = nullptr;
    cudaEvent_t* ev = nullptr;
    if (m.concurrent && m.side[0] && (int64_t)m.out_list.size() < kForkOut) {
        s1 = (cudaStream_t)m.side[0];
        s2 = (cudaStream_t)m.side[1];
        ev = (cudaEvent_t*)const_cast<Mesh&>(m).fork_ev;
    }
    if (precision == 0) {
        if (jv) launch_all<double, true>(m, A, s, nullptr, s1, s2, ev, generic); else launch_all<double, false>(m, A, s, nullptr, s1, s2, ev, generic);
    } else {
        if (jv) launch_all<float, true>(m, A, s, nullptr, s1, s2, ev); else launch_all<float, false>(m, A, s, nullptr, s1, s2, ev);
    }
    launch_strong_rows(m, A, ph, jv, s, true, precision);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

// one-time launch attributes of the element kernels (call before any stream capture)
void vms_prepare() {
    interior_blocks_per_sm<double, true>();
    interior_blocks_per_sm<double, false>();
    interior_blocks_per_sm<double, true, 2, true>();
    interior_blocks_per_sm<double, false, 2, true>();
    interior_blocks_per_sm<float, true>();
    interior_blocks_per_sm<float, false>();
    interior_blocks_per_sm<float, true, 5>();
    interior_blocks_per_sm<float, false, 5>();
}

int vms_apply(const Mesh& m, const double* u, const double* up, const double* up2, const double* f,
              const imga_physics& ph, int precision, const double* v, double* out, void* stream, bool generic) {
    return vms_apply_ws(m, u, up, up2, f, ph, precision, v, out, stream, nullptr, generic);
}

// ------------------------------------------------------------------------------------------
// J v with no allocation at all: the per-call node workspace lives in this fixed array, which
// every GPU that loads the library holds until the process exits.  Host code must not pass the
// array's name to a kernel (on the host it names a shadow, not device memory): its device
// address is looked up once per device with cudaGetSymbolAddress.
// ------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

static std::mutex g_noalloc_mu;
static void* g_noalloc_addr[kMaxDevices] = {};

int vms_jvp_noalloc(const Mesh& m, const double* u, const double* up, const double* up2, const double* f,
                    const imga_physics& ph, int precision, const double* v, double* out, void* stream,
                    std::string& err) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { err = "no usable current device"; return 1; }
    if (dev != m.device) { err = "the mesh's device must be current"; return 1; }
    const size_t next = (size_t)(m.n_nodes() + m.n_hang());
    const size_t per_node = (size_t)(f ? 20 : 16) * (precision == 0 ? sizeof(double) : sizeof(float));
    if (next * per_node > kNoAllocScratchBytes) {
        err = "mesh too large for the fixed scratch: needs " + std::to_string(next * per_node) + " bytes, limit " +
              std::to_string(kNoAllocScratchBytes);
        return 1;
    }
    void* ws = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_addr[dev]) {
            void* p = nullptr;
            cudaError_t rc = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (rc != cudaSuccess || !p) { err = std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(rc); return 1; }
            g_noalloc_addr[dev] = p;
        }
        ws = g_noalloc_addr[dev];
    }
    if (vms_apply_ws(m, u, up, up2, f, ph, precision, v, out, stream, ws, false)) { err = "launch failed"; return 1; }
    return 0;
}

// F [3] (device) = force of the fluid on the body at the state (u, u_prev); part: kForceBlocks x 3
// doubles of workspace
int surface_force(const Mesh& m, const double* u, const double* up, const imga_physics& ph, double* F, double* part,
                  void* stream) {
    cudaStream_t s = (cudaStream_t)stream;
    Args A = make_args(m, u, up, up, nullptr, ph, nullptr, nullptr);
    const int64_t next = m.n_nodes() + m.n_hang();
    double* ndv = node_workspace<double>(m, nullptr);
    A.ndv = ndv;
    A.ndt = ndv + 8 * next;
    A.ndf = nullptr;
    if (next > 0) launch_node_prep<double, false>(A, ndv, ndv + 8 * next, nullptr, s);
    const int64_t ns = (int64_t)m.sq.size() / 10;
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(kForceBlocks, (ns + 255) / 256));
    surface_force_partial<<<nb, 256, 0, s>>>(A, m.d.sq_elem, m.d.sq_x, m.d.sq_n, m.d.sq_w, m.d.sq_taub, ns, part);
    surface_force_final<<<1, 32, 0, s>>>(nb, part, F);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

void profile_reset(Mesh& m) {
    for (int k = 0; k < kProfKinds; ++k) {
        for (auto& p : m.prof_ev[k]) { cudaEventDestroy((cudaEvent_t)p.a); cudaEventDestroy((cudaEvent_t)p.b); }
        m.prof_ev[k].clear();
        m.prof_ms[k] = 0.0;
        m.prof_n[k] = 0;
    }
}

int profile_collect(Mesh& m) {
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    for (int k = 0; k < kProfKinds; ++k) {
        for (auto& p : m.prof_ev[k]) {
            float ms = 0.f;
            cudaEventElapsedTime(&ms, (cudaEvent_t)p.a, (cudaEvent_t)p.b);
            m.prof_ms[k] += ms;
            m.prof_n[k] += p.launches;
            cudaEventDestroy((cudaEvent_t)p.a);
            cudaEventDestroy((cudaEvent_t)p.b);
        }
        m.prof_ev[k].clear();
    }
    return 0;
}

}  // namespace imga
