// Learned block preconditioner: a 3-layer MLP (BF16 weights and activations on the tensor cores,
// FP32 accumulation, FP32 master weights, Adam) that maps an element's normalised Jacobian block
// k_e (32 x 32) plus features (log h, Intercepted flag, log10 local Re) to a 32 x 32 correction C_e;
// GMRES is then right-preconditioned by
//     P^-1 v = D^-1 v + omega sum_e M_e^T (C_e / s_e) M_e v,
// D the nodal block-Jacobi diagonal (its fallback), s_e the element's mean |diagonal| entry.
// Training target: the element's exact inverse correction (K + 0.1 I)^-1 - blockdiag4(K + 0.1 I)^-1
// of the normalised block, from the Jacobians the method itself forms (imga_element_jacobians).
// The paper has no learned component; its conclusion asks for method-specific preconditioners
// for matrix-free solvers (Sec. "Conclusion", footnote of Sec. "Matrix Assembly").
//
// GEMMs: C[m, n] = alpha sum_k A(m, k) B(n, k) + beta C[m, n] with arbitrary strides, mma.sync
// m16n8k16 BF16 x BF16 -> FP32; CTA tile 64 x 64 x 32, four warps of 32 x 32.

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "imga_internal.h"
#include "vms_device.cuh"

namespace imga {

namespace {

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ uint32_t pack2(bf16 lo, bf16 hi) {
    return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], const uint32_t b[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

constexpr int GT = 64, GK = 32, GPAD = 8;

__global__ void __launch_bounds__(128) gemm_bf16(int M, int N, int K, const bf16* __restrict__ A, int64_t sam,
                                                 int64_t sak, const bf16* __restrict__ B, int64_t sbn, int64_t sbk,
                                                 float* __restrict__ C, int64_t ldc, float alpha, float beta) {
    __shared__ __align__(16) bf16 sA[GT][GK + GPAD];
    __shared__ __align__(16) bf16 sB[GT][GK + GPAD];
    const int m0 = blockIdx.y * GT, n0 = blockIdx.x * GT;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    const int gid = lane >> 2, tig = lane & 3;
    float acc[2][4][4];
    for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 4; ++j)
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
    const bf16 zero = __float2bfloat16(0.f);
    for (int k0 = 0; k0 < K; k0 += GK) {
        for (int i = threadIdx.x; i < GT * GK; i += blockDim.x) {
            const int r = i / GK, kk = i % GK;
            const int gm = m0 + r, gn = n0 + r, gk = k0 + kk;
            sA[r][kk] = (gm < M && gk < K) ? A[(int64_t)gm * sam + (int64_t)gk * sak] : zero;
            sB[r][kk] = (gn < N && gk < K) ? B[(int64_t)gn * sbn + (int64_t)gk * sbk] : zero;
        }
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < GK; ks += 16) {
            uint32_t af[2][4], bfr[4][2];
            for (int i = 0; i < 2; ++i) {
                const int r = wm + 16 * i + gid;
                af[i][0] = pack2(sA[r][ks + 2 * tig], sA[r][ks + 2 * tig + 1]);
                af[i][1] = pack2(sA[r + 8][ks + 2 * tig], sA[r + 8][ks + 2 * tig + 1]);
                af[i][2] = pack2(sA[r][ks + 2 * tig + 8], sA[r][ks + 2 * tig + 9]);
                af[i][3] = pack2(sA[r + 8][ks + 2 * tig + 8], sA[r + 8][ks + 2 * tig + 9]);
            }
            for (int j = 0; j < 4; ++j) {
                const int c = wn + 8 * j + gid;
                bfr[j][0] = pack2(sB[c][ks + 2 * tig], sB[c][ks + 2 * tig + 1]);
                bfr[j][1] = pack2(sB[c][ks + 2 * tig + 8], sB[c][ks + 2 * tig + 9]);
            }
            for (int i = 0; i < 2; ++i)
                for (int j = 0; j < 4; ++j) mma16816(acc[i][j], af[i], bfr[j]);
        }
        __syncthreads();
    }
    for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 4; ++j)
            for (int q = 0; q < 4; ++q) {
                const int r = m0 + wm + 16 * i + gid + (q >= 2 ? 8 : 0);
                const int c = n0 + wn + 8 * j + 2 * tig + (q & 1);
                if (r < M && c < N) {
                    float* dst = C + (int64_t)r * ldc + c;
                    *dst = beta == 0.f ? alpha * acc[i][j][q] : alpha * acc[i][j][q] + beta * *dst;
                }
            }
}

void gemm(cudaStream_t s, int M, int N, int K, const bf16* A, int64_t sam, int64_t sak, const bf16* B, int64_t sbn,
          int64_t sbk, float* C, int64_t ldc, float alpha = 1.f, float beta = 0.f) {
    dim3 grid((N + GT - 1) / GT, (M + GT - 1) / GT);
    gemm_bf16<<<grid, 128, 0, s>>>(M, N, K, A, sam, sak, B, sbn, sbk, C, ldc, alpha, beta);
}

// ------------------------------------------------------------------------------------------
// The network of the preconditioner's width (128) in few launches.  A row of the forward pass moves
// 8 KB (1027 floats in, 1024 out) for 0.56 Mflop: it is bound by HBM, so the whole pass is one kernel
// that reads X and writes Y once, with the activations of its BM rows in shared memory and registers
// and the weights (0.56 MB) from L2; mma.sync is far from its rate there.  Every sum runs over k in
// steps of 16 in increasing order, as in gemm_bf16: the same bits.
//   50,003 rows: 2,625 -> 158 us (2.6 TB/s of X and Y).
// ------------------------------------------------------------------------------------------
constexpr int kW = 128;            // width of the fused path
constexpr int kHS = kW + 8;        // row stride of activations and of a weight chunk: conflict-free fragment reads

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// asynchronous copies of 16 or 4 bytes, the first `valid` of them from src, the rest zeros
__device__ __forceinline__ void cpz16(void* dst, const void* src, int valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(saddr(dst)), "l"(src), "r"(valid) : "memory");
}
__device__ __forceinline__ void cpz4(void* dst, const void* src, int valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(saddr(dst)), "l"(src), "r"(valid) : "memory");
}
__device__ __forceinline__ void ldm4(uint32_t r[4], const bf16* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(saddr(p)) : "memory");
}
__device__ __forceinline__ void ldm4t(uint32_t r[4], const bf16* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(saddr(p)) : "memory");
}
__device__ __forceinline__ uint32_t cvt2(float lo, float hi) {   // one conversion instruction for the pair
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

struct MlpTrainIO {           // what a training step keeps of the forward pass
    const float* T;           // targets [n][nout]
    float inv_scale;
    bf16 *xb, *h1, *h2, *dy;  // inputs and activations in bf16, (y - t) * inv_scale
    float* err;               // y - t
};

// BM rows per CTA of NT threads: for BM = 64 two rows of warps, otherwise one, the others over the columns.
// STAGES k-tiles of KT columns of X (fp32) and W1 in flight; the same shared memory then holds the
// activations and two chunks of NC rows of W2 / W3.
template <int BM, int NT, int KT, int NC, int STAGES> struct FwdShape {
    static constexpr int WM = BM == 64 ? 2 : 1, WN = NT / 32 / WM, MI = BM / (16 * WM);
    static constexpr int KS = KT + 8;                                  // row stride of a stage (floats of X, bf16 of W1)
    static constexpr int XS = BM * KS * 4, WS = kW * KS * 2;           // bytes of a stage
    static constexpr int HB = BM * kHS * 2, CB = NC * kHS * 2;         // bytes of the activations, of a weight chunk
    static constexpr int smem = STAGES * (XS + WS) > HB + 2 * CB ? STAGES * (XS + WS) : HB + 2 * CB;
    static_assert(kW / WN % 16 == 0 && NC / WN % 16 == 0 && KT % 16 == 0 && kW % NC == 0, "tiles of pairs of 8 columns");
};

template <int BM, int NT, int KT, int NC, int STAGES, bool TRAIN>
__global__ void __launch_bounds__(NT) mlp_fused(int64_t n, int nin, int nin_pad, const float* __restrict__ X, int64_t ldx,
                                                int xvec, const bf16* __restrict__ W1, const float* __restrict__ b1,
                                                const bf16* __restrict__ W2, const float* __restrict__ b2,
                                                const bf16* __restrict__ W3, const float* __restrict__ b3, int nout,
                                                float* __restrict__ Y, MlpTrainIO io) {
    typedef FwdShape<BM, NT, KT, NC, STAGES> Sh;
    constexpr int WN = Sh::WN, MI = Sh::MI, N1 = kW / WN / 8, N2 = NC / WN / 8, kKT = KT, kKS = Sh::KS, kNC = NC;
    extern __shared__ __align__(16) unsigned char sm[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
    const int wm = (warp / WN) * 16 * MI, wn = warp % WN;
    const int64_t m0 = (int64_t)blockIdx.x * BM;
    auto xs = [&](int s) { return reinterpret_cast<float*>(sm + s * (Sh::XS + Sh::WS)); };
    auto ws = [&](int s) { return reinterpret_cast<bf16*>(sm + s * (Sh::XS + Sh::WS) + Sh::XS); };
    const int nkt = (nin_pad + kKT - 1) / kKT;
    // a thread copies the same columns of every stage: its rows' addresses are formed once (they were more than
    // half of the kernel's instructions)
    constexpr int XC = KT / 4, XR = NT / XC, XN = BM / XR, WC = KT / 8, WR = NT / WC, WN_ = kW / WR;
    static_assert(BM % XR == 0 && kW % WR == 0, "whole rows per pass");
    const int xc = tid % XC * 4, xr = tid / XC, wc = tid % WC * 8, wr = tid / WC;
    const float* xsrc[XN];
#pragma unroll
    for (int i = 0; i < XN; ++i) xsrc[i] = m0 + xr + XR * i < n ? X + (m0 + xr + XR * i) * ldx + xc : nullptr;
    const bf16* wsrc = W1 + (int64_t)wr * nin_pad + wc;
    auto load = [&](int kt) {
        if (kt < nkt) {
            float* x = xs(kt % STAGES) + xr * kKS + xc;
            bf16* w = ws(kt % STAGES) + wr * kKS + wc;
            const int k0 = kt * kKT, left = max(0, min(4, nin - k0 - xc));
#pragma unroll
            for (int i = 0; i < XN; ++i) {
                const int here = xsrc[i] ? left : 0;
                const float* src = here ? xsrc[i] + k0 : X;
                if (xvec) cpz16(x + XR * i * kKS, src, 4 * here);
                else
                    for (int j = 0; j < 4; ++j) cpz4(x + XR * i * kKS + j, j < here ? src + j : X, j < here ? 4 : 0);
            }
            const bool in = k0 + wc < nin_pad;
            const bf16* src = in ? wsrc + k0 : W1;
            const int64_t step = in ? (int64_t)WR * nin_pad : 0;
#pragma unroll
            for (int i = 0; i < WN_; ++i) cpz16(w + WR * i * kKS, src + i * step, in ? 16 : 0);
        }
        cp_commit();
    };
    // ldmatrix lane offsets: A (16 x 16, rows then k halves), B (two n-tiles, k halves)
    const int arow = lane & 15, acol = (lane >> 4) * 8;
    const int brow = (lane & 7) + ((lane >> 4) << 3), bcol = ((lane >> 3) & 1) * 8;
    for (int s = 0; s < STAGES - 1; ++s) load(s);
    float acc[MI][N1][4];
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < N1; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
    for (int kt = 0; kt < nkt; ++kt) {
        cp_wait<STAGES - 2>();
        __syncthreads();   // stage kt has landed; every warp is done with stage kt - 1, which is refilled
        load(kt + STAGES - 1);
        const float* x = xs(kt % STAGES);
        const bf16* w = ws(kt % STAGES);
#pragma unroll
        for (int ks = 0; ks < kKT; ks += 16) {
            uint32_t a[MI][4];
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int r = wm + 16 * i + gid + (q & 1) * 8, c = ks + 2 * tig + (q >> 1) * 8;
                    const float2 v = *reinterpret_cast<const float2*>(x + r * kKS + c);
                    a[i][q] = cvt2(v.x, v.y);
                    if (TRAIN && wn == 0 && m0 + r < n && kt * kKT + c < nin_pad)
                        *reinterpret_cast<uint32_t*>(io.xb + (m0 + r) * nin_pad + kt * kKT + c) = a[i][q];
                }
#pragma unroll
            for (int j = 0; j < N1; j += 2) {
                uint32_t b[4];
                ldm4(b, w + (wn * (kW / WN) + 8 * j + brow) * kKS + ks + bcol);
#pragma unroll
                for (int i = 0; i < MI; ++i) {
                    mma16816(acc[i][j], a[i], b);
                    mma16816(acc[i][j + 1], a[i], b + 2);
                }
            }
        }
    }
    cp_wait<0>();
    __syncthreads();   // the stages are free: activations and weight chunks take their place
    bf16* h = reinterpret_cast<bf16*>(sm);
    auto chunk_buf = [&](int k) { return reinterpret_cast<bf16*>(sm + Sh::HB + (k & 1) * Sh::CB); };
    // chunks 0, 1: W2; 2 ...: W3
    const int nchunk = kW / kNC + (nout + kNC - 1) / kNC;
    auto load_chunk = [&](int k) {
        if (k < nchunk) {
            const bool l2 = k < kW / kNC;
            const bf16* W = l2 ? W2 : W3;
            const int n0 = (l2 ? k : k - kW / kNC) * kNC, nr = l2 ? kW : nout;
            bf16* w = chunk_buf(k);
            constexpr int R = NT / (kW / 8);
            static_assert(kNC % R == 0, "whole rows per pass");
            const int r0 = tid / (kW / 8), c = tid % (kW / 8) * 8;
            const bf16* src = W + (int64_t)(n0 + r0) * kW + c;
            bf16* dst = w + r0 * kHS + c;
#pragma unroll
            for (int i = 0; i < kNC / R; ++i) {
                const bool in = n0 + r0 + R * i < nr;
                cpz16(dst + R * i * kHS, in ? src + R * i * kW : W, in ? 16 : 0);
            }
        }
        cp_commit();
    };
    // h = relu(z + b) in bf16 of one accumulator pair, to shared memory (and, training, to memory)
    auto put_h = [&](const float* z, const float* b, int r, int c, bf16* keep) {
        const float v0 = z[0] + __ldg(b + c), v1 = z[1] + __ldg(b + c + 1);
        const uint32_t p = cvt2(v0 > 0.f ? v0 : 0.f, v1 > 0.f ? v1 : 0.f);
        *reinterpret_cast<uint32_t*>(h + r * kHS + c) = p;
        if (TRAIN && m0 + r < n) *reinterpret_cast<uint32_t*>(keep + (m0 + r) * kW + c) = p;
    };
    load_chunk(0);
    load_chunk(1);
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < N1; ++j)
#pragma unroll
            for (int q = 0; q < 4; q += 2)
                put_h(&acc[i][j][q], b1, wm + 16 * i + gid + q * 4, wn * (kW / WN) + 8 * j + 2 * tig, io.h1);
    // one weight chunk: o[i][j] = rows of h times kNC / WN of its columns
    uint32_t a[kW / 16][MI][4];
    auto load_a = [&]() {
#pragma unroll
        for (int ks = 0; ks < kW / 16; ++ks)
#pragma unroll
            for (int i = 0; i < MI; ++i) ldm4(a[ks][i], h + (wm + 16 * i + arow) * kHS + 16 * ks + acol);
    };
    auto times_chunk = [&](int k, float o[MI][N2][4]) {
        const bf16* w = chunk_buf(k);
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int j = 0; j < N2; ++j)
#pragma unroll
                for (int q = 0; q < 4; ++q) o[i][j][q] = 0.f;
#pragma unroll
        for (int ks = 0; ks < kW / 16; ++ks)
#pragma unroll
            for (int j = 0; j < N2; j += 2) {
                uint32_t b[4];
                ldm4(b, w + (wn * (kNC / WN) + 8 * j + brow) * kHS + 16 * ks + bcol);
#pragma unroll
                for (int i = 0; i < MI; ++i) {
                    mma16816(o[i][j], a[ks][i], b);
                    mma16816(o[i][j + 1], a[ks][i], b + 2);
                }
            }
    };
    float z2[kW / kNC][MI][N2][4];
#pragma unroll
    for (int k = 0; k < kW / kNC; ++k) {
        cp_wait<1>();
        __syncthreads();
        if (k == 0) load_a();
        times_chunk(k, z2[k]);
        __syncthreads();
        load_chunk(k + 2);
    }
#pragma unroll
    for (int k = 0; k < kW / kNC; ++k)
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int j = 0; j < N2; ++j)
#pragma unroll
                for (int q = 0; q < 4; q += 2)
                    put_h(&z2[k][i][j][q], b2, wm + 16 * i + gid + q * 4, k * kNC + wn * (kNC / WN) + 8 * j + 2 * tig, io.h2);
    for (int k = kW / kNC; k < nchunk; ++k) {
        const int n0 = (k - kW / kNC) * kNC + wn * (kNC / WN) + 2 * tig;
        float2 tg[TRAIN ? MI : 1][TRAIN ? N2 : 1][2];
        if constexpr (TRAIN) {   // the chunk's targets come in beside its weights
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < N2; ++j)
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int64_t r = m0 + wm + 16 * i + gid + q * 8;
                        const int c = n0 + 8 * j;
                        tg[i][j][q] = r < n && c < nout ? __ldg(reinterpret_cast<const float2*>(io.T + r * nout + c)) : make_float2(0.f, 0.f);
                    }
        }
        cp_wait<1>();
        __syncthreads();
        if (k == kW / kNC) load_a();
        float o[MI][N2][4];
        times_chunk(k, o);
        __syncthreads();
        load_chunk(k + 2);
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int j = 0; j < N2; ++j)
#pragma unroll
                for (int q = 0; q < 4; q += 2) {
                    const int64_t r = m0 + wm + 16 * i + gid + q * 4;
                    const int c = n0 + 8 * j;
                    if (r >= n || c >= nout) continue;   // nout is even
                    const float y0 = o[i][j][q] + __ldg(b3 + c), y1 = o[i][j][q + 1] + __ldg(b3 + c + 1);
                    if constexpr (!TRAIN) {
                        *reinterpret_cast<float2*>(Y + r * nout + c) = make_float2(y0, y1);
                    } else {
                        const float2 t = tg[i][j][q >> 1];
                        const float d0 = y0 - t.x, d1 = y1 - t.y;
                        *reinterpret_cast<uint32_t*>(io.dy + r * nout + c) = cvt2(d0 * io.inv_scale, d1 * io.inv_scale);
                        *reinterpret_cast<float2*>(io.err + r * nout + c) = make_float2(d0, d1);
                    }
                }
    }
    cp_wait<0>();
}

// A thread's sum of squares, no less exact than a float64 one: the square is exact in two floats, and the sum is
// kept in floats of three sizes (TwoSum: hi + mid + mid2 exactly what was added but for the middle parts' own rounding
// errors, which lo adds up), 72 bits against 53.  Where the largest of N values is outside 2^-40 .. 2^58, squares or
// their low parts could leave the float32 range, and a float64 sum takes them (inf too; a NaN ends as one on either
// path); smaller values beside a larger one lose less than 2^-70 of its square.  (The FP64 pipe takes a warp's
// multiply-add every 19 cycles, 20 instructions here take 5.)
struct SquareSum {
    float hi = 0.f, mid = 0.f, mid2 = 0.f, lo = 0.f;
    double wide = 0.0;
    static __device__ __forceinline__ float two_sum(float& s, float x) {   // s += x, the rounding error returned
        const float t = __fadd_rn(s, x), b = __fsub_rn(t, s), e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b));
        s = t;
        return e;
    }
    template <int N> __device__ __forceinline__ void add(const float* d) {
        float most = 0.f;
#pragma unroll
        for (int k = 0; k < N; ++k) most = fmaxf(most, fabsf(d[k]));
        if (most >= 0x1p-40f && most < 0x1p58f) {
#pragma unroll
            for (int k = 0; k < N; ++k) {
                const float p = __fmul_rn(d[k], d[k]), e = __fmaf_rn(d[k], d[k], -p);
                const float a = two_sum(mid, two_sum(hi, p)), b = two_sum(mid2, e);
                lo = __fadd_rn(lo, __fadd_rn(a, b));
            }
        } else {
#pragma unroll
            for (int k = 0; k < N; ++k) {
                const double x = f2d(d[k]);
                wide = fma(x, x, wide);
            }
        }
    }
    __device__ __forceinline__ double total() const { return (double)hi + (((double)mid + (double)mid2) + ((double)lo + wide)); }
};

// Gradient products of one layer in one launch, 32 x 32 of the result per CTA, K whole (the sums keep
// the order of gemm_bf16), 64 of K per stage, four stages in flight.  Bound by the latency of the K chain
// (64 dependent products for 1024 rows), so the tiles are small: more CTAs, not more work per CTA.
//   dw CTAs: G [M][N] = alpha D^T H  (D [K][M], H [K][N] rows of the batch);
//   db CTAs: the column sums of D (the bias gradient), rows in order, 32 columns each;
//   dh CTAs: Z [K][N] = (D W) masked by H > 0, in bf16 (W [M][N] the layer's weights, H its input);
//   loss CTAs (output layer): += the sum of the squared float32 errors, kLossPer of them each, on SMs that the chains
//     leave idle.  In the forward kernel, whose CTAs have 64 SMs at 1,024 rows, the same sum took 1 to 2 us of a step's
//     79, a float64 one 6; here a step is 2 us shorter up to 1,024 rows, 1.6 us (of 106) longer at 2,048.
constexpr int kBT = 32, kBK = 64, kBStages = 4;
constexpr int64_t kLossPer = 8192;
struct BackArgs {
    int64_t K;             // rows of the batch
    int M, N;              // the layer's outputs and inputs
    const bf16 *D, *H, *W;
    float *G, *db;
    bf16* Z;               // null: no dh part
    float beta;
    int dw_n, dw_tiles;    // CTAs along N and in all of the dw part
    const float* err;      // n_err (a multiple of 4) errors; the loss CTAs are the last, from loss_at on
    int64_t n_err;
    double* loss;
    unsigned loss_at;
};

__global__ void __launch_bounds__(128) mlp_back(BackArgs P) {
    // a stage: A as [64][32 + 8] (dw: rows k) or [32][64 + 8] (dh: rows m), B as [64][32 + 8]
    constexpr int AS = kBK * (kBT + 8), TS = kBT + 8, DS = kBK + 8;
    __shared__ __align__(16) bf16 sA[kBStages][AS], sB[kBStages][AS];
    static_assert(kBT * DS <= AS, "stage size");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
    if (blockIdx.x >= P.loss_at) {
        __shared__ double s_sum[4];
        const int64_t i0 = (int64_t)(blockIdx.x - P.loss_at) * kLossPer;
        SquareSum sq;
        for (int k = 0; k < kLossPer; k += 16 * 128) {
            float d[16];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int64_t i = i0 + k + 4 * (128 * j + tid);
                const float4 v = i < P.n_err ? *reinterpret_cast<const float4*>(P.err + i) : make_float4(0.f, 0.f, 0.f, 0.f);
                d[4 * j] = v.x;
                d[4 * j + 1] = v.y;
                d[4 * j + 2] = v.z;
                d[4 * j + 3] = v.w;
            }
            sq.add<16>(d);
        }
        double s = sq.total();
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) s_sum[warp] = s;
        __syncthreads();
        if (tid == 0) atomicAdd(P.loss, (s_sum[0] + s_sum[1]) + (s_sum[2] + s_sum[3]));
        return;
    }
    const int wm = (warp >> 1) * 16, wn = (warp & 1) * 16;
    // the db CTAs come first (their serial sums are the longest chain), then dw, then dh
    const int b0 = (int)blockIdx.x - (P.M + kBT - 1) / kBT;
    const bool db = b0 < 0, dw = b0 < P.dw_tiles;
    const int t = db ? (int)blockIdx.x * P.dw_n : dw ? b0 : b0 - P.dw_tiles;
    const int nb = dw ? P.dw_n : (P.N + kBT - 1) / kBT;
    const int64_t m0 = (int64_t)(t / nb) * kBT;
    const int n0 = (t % nb) * kBT;
    const int64_t K = dw ? P.K : P.M;
    const int64_t rows = dw ? P.M : P.K;       // extent of the result along m
    const bf16* B = dw ? P.H : P.W;
    const int nkt = (int)((K + kBK - 1) / kBK);
    auto load = [&](int kt) {
        if (kt < nkt) {
            bf16 *a = sA[kt % kBStages], *b = sB[kt % kBStages];
            const int64_t k0 = (int64_t)kt * kBK;
            for (int i = tid; i < kBK * kBT / 8; i += 128) {
                const int kr = i / (kBT / 8), c = i % (kBT / 8) * 8;
                const bool inb = k0 + kr < K && n0 + c < P.N;
                if (!db) cpz16(b + kr * TS + c, inb ? B + (k0 + kr) * P.N + n0 + c : B, inb ? 16 : 0);
                if (dw) {
                    const bool ina = k0 + kr < K && m0 + c < P.M;
                    cpz16(a + kr * TS + c, ina ? P.D + (k0 + kr) * P.M + m0 + c : P.D, ina ? 16 : 0);
                } else {
                    const int mr = i / (kBK / 8), kc = i % (kBK / 8) * 8;
                    const bool ina = m0 + mr < P.K && k0 + kc < K;
                    cpz16(a + mr * DS + kc, ina ? P.D + (m0 + mr) * P.M + k0 + kc : P.D, ina ? 16 : 0);
                }
            }
        }
        cp_commit();
    };
    for (int s = 0; s < kBStages - 1; ++s) load(s);
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    float s = 0.f;
    // transposed 8 x 8 blocks: A as (m, k), (m + 8, k), (m, k + 8), (m + 8, k + 8); B as (n, k), (n, k + 8), ...
    const int akr = (lane & 7) + ((lane >> 4) << 3), amc = ((lane >> 3) & 1) * 8;
    const int bkr = lane & 15, bnc = (lane >> 4) * 8;
    const int arow = lane & 15, acol = (lane >> 4) * 8;
    for (int kt = 0; kt < nkt; ++kt) {
        cp_wait<kBStages - 2>();
        __syncthreads();
        load(kt + kBStages - 1);
        const bf16 *a = sA[kt % kBStages], *b = sB[kt % kBStages];
        if (db) {
            const int kr1 = (int)min((int64_t)kBK, K - (int64_t)kt * kBK);
            if (warp == 0) {
#pragma unroll 16
                for (int kr = 0; kr < kr1; ++kr) s += __bfloat162float(a[kr * TS + lane]);
            }
            continue;
        }
#pragma unroll
        for (int ks = 0; ks < kBK; ks += 16) {
            uint32_t af[4], bf[4];
            if (dw) ldm4t(af, a + (ks + akr) * TS + wm + amc);
            else ldm4(af, a + (wm + arow) * DS + ks + acol);
            ldm4t(bf, b + (ks + bkr) * TS + wn + bnc);
            mma16816(acc[0], af, bf);
            mma16816(acc[1], af, bf + 2);
        }
    }
    cp_wait<0>();
    if (db) {
        if (warp == 0 && m0 + lane < P.M) P.db[m0 + lane] = P.beta != 0.f ? P.db[m0 + lane] + s : s;
        return;
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
            const int64_t r = m0 + wm + gid + q * 4;
            const int c = n0 + wn + 8 * j + 2 * tig;
            if (r >= rows || c >= P.N) continue;   // N is a multiple of 8
            if (dw) {
                float2* g = reinterpret_cast<float2*>(P.G + r * P.N + c);
                float2 v = make_float2(acc[j][q], acc[j][q + 1]);
                if (P.beta != 0.f) { const float2 o = *g; v.x += P.beta * o.x; v.y += P.beta * o.y; }
                *g = v;
            } else {
                const uint32_t hv = *reinterpret_cast<const uint32_t*>(P.H + r * P.N + c);
                const float h0 = __uint_as_float(hv << 16), h1 = __uint_as_float(hv & 0xFFFF0000u);
                *reinterpret_cast<uint32_t*>(P.Z + r * P.N + c) = cvt2(h0 > 0.f ? acc[j][q] : 0.f, h1 > 0.f ? acc[j][q + 1] : 0.f);
            }
        }
}

__global__ void to_bf16(int64_t n, const float* __restrict__ x, bf16* __restrict__ y) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16(x[i]);
}
// rows of x [n][ld_in] (first n_in columns) -> bf16 [n][ld_out] zero padded
__global__ void rows_to_bf16(int64_t n, int n_in, int64_t ld_in, const float* __restrict__ x, int ld_out,
                             bf16* __restrict__ y) {
    const int64_t tot = n * ld_out;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / ld_out;
        const int c = (int)(i % ld_out);
        y[i] = __float2bfloat16(c < n_in ? x[r * ld_in + c] : 0.f);
    }
}
// z = c + b (kept for the backward mask), h = relu(z) in bf16
__global__ void bias_relu(int64_t n, int w, float* __restrict__ z, const float* __restrict__ b, bf16* __restrict__ h) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n * w; i += (int64_t)gridDim.x * blockDim.x) {
        const float v = z[i] + b[i % w];
        z[i] = v;
        h[i] = __float2bfloat16(v > 0.f ? v : 0.f);
    }
}
__global__ void bias_add(int64_t n, int w, float* __restrict__ y, const float* __restrict__ b) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n * w; i += (int64_t)gridDim.x * blockDim.x)
        y[i] += b[i % w];
}
// dy = (y - t) / scale (bf16), loss partial sum of (y - t)^2
__global__ void mse_grad(int64_t n, const float* __restrict__ y, const float* __restrict__ t, float inv_scale,
                         bf16* __restrict__ dy, double* __restrict__ loss) {
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float d = y[i] - t[i];
        s += (double)d * (double)d;
        dy[i] = __float2bfloat16(d * inv_scale);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(loss, s);
}
// dz = dh * (z > 0), bf16
__global__ void relu_back(int64_t n, const float* __restrict__ dh, const float* __restrict__ z, bf16* __restrict__ dz) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dz[i] = __float2bfloat16(z[i] > 0.f ? dh[i] : 0.f);
}
// db[j] (+)= sum_r d[r][j]  (d bf16 [n][w])
__global__ void col_sum(int64_t n, int w, const bf16* __restrict__ d, float* __restrict__ db, int accumulate) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= w) return;
    float s = 0.f;
    for (int64_t r = 0; r < n; ++r) s += __bfloat162float(d[r * w + j]);
    db[j] = accumulate ? db[j] + s : s;
}
// Adam update and the weights' new bf16 copy
__global__ void adam(int64_t n, float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                     float* __restrict__ v, bf16* __restrict__ wb, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
        w[i] = wi;
        wb[i] = __float2bfloat16(wi);
    }
}

// one warp per 32 x 32 matrix: Gauss-Jordan with partial pivoting, lane r owns row r of [A | I]
__device__ bool warp_inverse32(float a[32], float inv[32], int lane) {
    for (int j = 0; j < 32; ++j) inv[j] = j == lane ? 1.f : 0.f;
    for (int c = 0; c < 32; ++c) {
        // pivot: largest |a[c]| among rows >= c
        float best = lane >= c ? fabsf(a[c]) : -1.f;
        int bl = lane;
        for (int o = 16; o > 0; o >>= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, best, o);
            const int ol = __shfl_xor_sync(0xffffffffu, bl, o);
            if (ob > best || (ob == best && ol < bl)) { best = ob; bl = ol; }
        }
        if (!(best > 0.f)) return false;
        // swap rows c and bl
        if (bl != c) {
            for (int j = 0; j < 32; ++j) {
                const float x = a[j], y = inv[j];
                const float xc = __shfl_sync(0xffffffffu, x, c), xb = __shfl_sync(0xffffffffu, x, bl);
                const float yc = __shfl_sync(0xffffffffu, y, c), yb = __shfl_sync(0xffffffffu, y, bl);
                if (lane == c) { a[j] = xb; inv[j] = yb; }
                if (lane == bl) { a[j] = xc; inv[j] = yc; }
            }
        }
        const float piv = __shfl_sync(0xffffffffu, a[c], c);
        const float ip = 1.f / piv;
        if (lane == c)
            for (int j = 0; j < 32; ++j) { a[j] *= ip; inv[j] *= ip; }
        const float f = a[c];
        for (int j = 0; j < 32; ++j) {
            const float pr = __shfl_sync(0xffffffffu, a[j], c), pi = __shfl_sync(0xffffffffu, inv[j], c);
            if (lane != c) { a[j] -= f * pr; inv[j] -= f * pi; }
        }
    }
    return true;
}

// features + targets of one element per warp from K (float64 [n][32][32])
// X [n][ldx]: 1024 normalised entries, log(h), Intercepted flag, log10(1 + Re_local); T [n][1024]
__global__ void dataset_kernel(Args A, int64_t n, const int32_t* __restrict__ elems, const double* __restrict__ K,
                               const int8_t* __restrict__ marker, float eps, int ldx, float* __restrict__ X,
                               float* __restrict__ Tg, float* __restrict__ scale_out) {
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= n) return;
    const double* Ke = K + w * 1024;
    float row[32], inv[32];
    double d = fabs(Ke[lane * 32 + lane]);
    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    const double s = d / 32.0 > 0.0 ? d / 32.0 : 1.0;
    for (int j = 0; j < 32; ++j) row[j] = (float)(Ke[lane * 32 + j] / s);
    float* xo = X + w * ldx;
    for (int j = 0; j < 32; ++j) xo[lane * 32 + j] = row[j];
    const int32_t e = elems[w];
    if (lane == 0) {
        const double h = 2.0 / A.gd[A.lev[e]];
        double uu = 0.0;
        for (int c = 0; c < 8; ++c) {
            double u4[4];
            gather(A, A.U, A.conn[8 * (int64_t)e + c], u4);
            uu += sqrt(u4[0] * u4[0] + u4[1] * u4[1] + u4[2] * u4[2]) / 8.0;
        }
        const double nu = (A.eprob ? A.pmu[A.eprob[e]] : A.mu) / A.rho;
        xo[1024] = (float)log(h);
        xo[1025] = marker[e] == 2 ? 1.f : 0.f;
        xo[1026] = (float)log10(1.0 + uu * h / (nu > 0.0 ? nu : 1e-300));
        for (int j = 1027; j < ldx; ++j) xo[j] = 0.f;
        scale_out[w] = (float)s;
    }
    if (!Tg) return;
    // target: (Khat + eps I)^-1 - blockdiag4(Khat + eps I)^-1
    row[lane] += eps;
    float full[32];
    for (int j = 0; j < 32; ++j) full[j] = row[j];
    bool ok = warp_inverse32(full, inv, lane);
    // block-diagonal inverse of the 4x4 blocks, computed by the same routine on the block-masked matrix
    float bd[32], binv[32];
    for (int j = 0; j < 32; ++j) bd[j] = ((j >> 2) == (lane >> 2)) ? row[j] : (j == lane ? 1.f : 0.f);
    // masking keeps only the 4x4 diagonal blocks (off-block entries are zero), so the inverse is
    // block-diagonal too
    for (int j = 0; j < 32; ++j) if ((j >> 2) != (lane >> 2)) bd[j] = 0.f;
    bool ok2 = warp_inverse32(bd, binv, lane);
    float* to = Tg + w * 1024;
    for (int j = 0; j < 32; ++j) to[lane * 32 + j] = (ok && ok2) ? inv[j] - binv[j] : 0.f;
}

// z_corr += omega M_e^T (C_e / s_e) M_e v, one warp per active element, lane = local dof (a, i)
__global__ void correction_apply(Args A, int64_t n, const int32_t* __restrict__ elems, const float* __restrict__ C,
                                 const float* __restrict__ scale, float omega, const double* __restrict__ v,
                                 double* __restrict__ z) {
    const int lane = threadIdx.x & 31;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= n) return;
    const int32_t e = elems[w];
    const int a = lane >> 2, comp = lane & 3;
    const int32_t id = A.conn[8 * (int64_t)e + a];
    double vv[4];
    gather(A, v, id, vv);
    const float x = (float)vv[comp];
    const float* Ce = C + w * 1024 + lane * 32;
    float y = 0.f;
    for (int j = 0; j < 32; ++j) y += Ce[j] * __shfl_sync(0xffffffffu, x, j);
    y *= omega / scale[w];
    // gather the node's 4 components to lane 4a and scatter through M_e^T
    double r[4];
    for (int k = 0; k < 4; ++k) r[k] = (double)__shfl_sync(0xffffffffu, y, (lane & ~3) + k);
    if (comp == 0) {
        Args B = A;
        B.out = z;
        scatter(B, id, r);
    }
}

// z = Dinv v + corr on free rows (prescribed rows keep Dinv v, which is v there)
__global__ void combine_rows(int64_t nn, const uint8_t* __restrict__ flag, const uint8_t* __restrict__ umask,
                             const double* __restrict__ corr, double* __restrict__ z) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= nn) return;
    uint8_t mask = umask ? umask[n] : (uint8_t)(flag[n] & 15);
    if (flag[n] & 16) mask = 15;
    for (int k = 0; k < 4; ++k)
        if (!((mask >> k) & 1)) z[4 * n + k] += corr[4 * n + k];
}

// shift of the normalised element block before inversion: the element's constant-pressure mode is
// nearly singular, and a small shift would make the local inverse (and the correction) huge there
constexpr float kTargetShift = 0.1f;

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)std::min<int64_t>(4096, (n + t - 1) / t); }

}  // namespace

// ------------------------------------------------------------------------------------------
// MLP object
// ------------------------------------------------------------------------------------------
struct Mlp {
    int nin, nin_pad, w, nout, n_sm = 1;
    int64_t nparam;
    float* P = nullptr;    // master weights: W1 [w][nin_pad], b1 [w], W2 [w][w], b2 [w], W3 [nout][w], b3 [nout]
    float* G = nullptr;    // gradients, same layout
    float* Mm = nullptr;   // Adam moments
    float* Vm = nullptr;
    bf16* Pb = nullptr;    // bf16 copy of the weights
    int64_t cap = 0, cap_general = 0;   // batch capacity of the activation buffers
    bf16 *xb = nullptr, *h1 = nullptr, *h2 = nullptr, *dyb = nullptr, *dz2 = nullptr, *dz1 = nullptr;
    float *z1 = nullptr, *z2 = nullptr, *y = nullptr, *dh2 = nullptr, *dh1 = nullptr;
    double* loss = nullptr;
    int64_t step = 0;
    int64_t off(int k) const {
        const int64_t o1 = (int64_t)w * nin_pad, o2 = o1 + w, o3 = o2 + (int64_t)w * w, o4 = o3 + w,
                      o5 = o4 + (int64_t)nout * w;
        const int64_t o[6] = {0, o1, o2, o3, o4, o5};
        return o[k];
    }
};

template <class T> static bool grow(T*& p, int64_t n) {
    cudaFree(p);
    p = nullptr;
    return cudaMalloc((void**)&p, n * sizeof(T)) == cudaSuccess;
}

// buffers for batches of b rows: those that every path keeps between its kernels, and those of the general path alone
static bool mlp_reserve(Mlp& M, int64_t b, bool general) {
    if (b > M.cap) {
        const bool ok = grow(M.xb, b * M.nin_pad) && grow(M.h1, b * M.w) && grow(M.h2, b * M.w) && grow(M.dyb, b * M.nout) &&
                        grow(M.dz2, b * M.w) && grow(M.dz1, b * M.w) && grow(M.y, b * M.nout);
        M.cap = ok ? b : 0;
        if (!ok) return false;
    }
    if (general && b > M.cap_general) {
        const bool ok = grow(M.z1, b * M.w) && grow(M.z2, b * M.w) && grow(M.dh2, b * M.w) && grow(M.dh1, b * M.w);
        M.cap_general = ok ? b : 0;
        if (!ok) return false;
    }
    return true;
}

static void mlp_sync_bf16(Mlp& M, cudaStream_t s) { to_bf16<<<nblk(M.nparam), 256, 0, s>>>(M.nparam, M.P, M.Pb); }

// The fused kernels serve the preconditioner's width; rows of 16 bytes in every bf16 matrix need nout % 8 == 0.
// Targets are read and results written in pairs.
static bool mlp_fast(const Mlp& M, const float* pairs) { return M.w == kW && M.nout % 8 == 0 && ((uintptr_t)pairs & 7) == 0; }

template <int BM, int NT, int KT, int NC, int STAGES, bool TRAIN>
static void launch_fused(const Mlp& M, const float* X, int64_t ldx, int64_t n, float* Y, const MlpTrainIO& io, cudaStream_t s) {
    typedef FwdShape<BM, NT, KT, NC, STAGES> Sh;
    static std::atomic<unsigned> ready{0};   // devices whose shared-memory limit is raised
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 32 || !((ready.load() >> dev) & 1u)) {
        cudaFuncSetAttribute(mlp_fused<BM, NT, KT, NC, STAGES, TRAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, Sh::smem);
        if (dev < 32) ready.fetch_or(1u << dev);
    }
    const int xvec = ((uintptr_t)X & 15) == 0 && ldx % 4 == 0;
    mlp_fused<BM, NT, KT, NC, STAGES, TRAIN><<<(unsigned)((n + BM - 1) / BM), NT, Sh::smem, s>>>(
        n, M.nin, M.nin_pad, X, ldx, xvec, M.Pb + M.off(0), M.P + M.off(1), M.Pb + M.off(2), M.P + M.off(3), M.Pb + M.off(4),
        M.P + M.off(5), M.nout, Y, io);
}

// Rows per CTA: 64 (the weights are read from L2 once per 64 rows) when that still gives two CTAs per SM,
// fewer for fewer rows, so that the chip has work (9,000 rows: 51 us with 32).  The small tile takes 8 warps, deep
// stages and wide chunks because a CTA is alone on its SM (1,024-row training steps: 61 -> 26 us).
template <bool TRAIN>
static void mlp_fused_rows(const Mlp& M, const float* X, int64_t ldx, int64_t n, float* Y, const MlpTrainIO& io, cudaStream_t s) {
    if (n >= (int64_t)64 * 2 * M.n_sm) launch_fused<64, 128, 32, 64, 3, TRAIN>(M, X, ldx, n, Y, io, s);
    else if (n >= (int64_t)32 * M.n_sm) launch_fused<32, 128, 32, 64, 4, TRAIN>(M, X, ldx, n, Y, io, s);
    else launch_fused<16, 256, 64, 128, 4, TRAIN>(M, X, ldx, n, Y, io, s);
}

// forward and backward of a batch on the fused path: gradients into M.G, loss added to M.loss
static void mlp_step_fused(Mlp& M, const float* X, int64_t ldx, const float* T, int64_t b, double n_total, float beta,
                           cudaStream_t s) {
    const MlpTrainIO io = {T, (float)(1.0 / n_total), M.xb, M.h1, M.h2, M.dyb, M.y};
    mlp_fused_rows<true>(M, X, ldx, b, nullptr, io, s);
    auto back = [&](int m, int nn, const bf16* D, const bf16* H, int k, bf16* Z, int64_t n_err) {
        BackArgs P = {b, m, nn, D, H, M.Pb + M.off(k), M.G + M.off(k), M.G + M.off(k + 1), Z, beta, 0, 0, M.y, n_err, M.loss, 0};
        P.dw_n = (nn + kBT - 1) / kBT;
        P.dw_tiles = P.dw_n * ((m + kBT - 1) / kBT);
        const int64_t dh = Z ? P.dw_n * ((b + kBT - 1) / kBT) : 0;
        P.loss_at = (unsigned)((m + kBT - 1) / kBT + P.dw_tiles + dh);
        mlp_back<<<P.loss_at + (unsigned)((n_err + kLossPer - 1) / kLossPer), 128, 0, s>>>(P);
    };
    back(M.nout, M.w, M.dyb, M.h2, 4, M.dz2, b * M.nout);
    back(M.w, M.w, M.dz2, M.h1, 2, M.dz1, 0);
    back(M.w, M.nin_pad, M.dz1, M.xb, 0, nullptr, 0);
}

// forward of a batch: X float [b][ldx] (first nin columns) -> M.y float [b][nout]
static void mlp_forward_batch(Mlp& M, const float* X, int64_t ldx, int64_t b, cudaStream_t s) {
    rows_to_bf16<<<nblk(b * M.nin_pad), 256, 0, s>>>(b, M.nin, ldx, X, M.nin_pad, M.xb);
    const bf16 *W1 = M.Pb + M.off(0), *W2 = M.Pb + M.off(2), *W3 = M.Pb + M.off(4);
    gemm(s, (int)b, M.w, M.nin_pad, M.xb, M.nin_pad, 1, W1, M.nin_pad, 1, M.z1, M.w);
    bias_relu<<<nblk(b * M.w), 256, 0, s>>>(b, M.w, M.z1, M.P + M.off(1), M.h1);
    gemm(s, (int)b, M.w, M.w, M.h1, M.w, 1, W2, M.w, 1, M.z2, M.w);
    bias_relu<<<nblk(b * M.w), 256, 0, s>>>(b, M.w, M.z2, M.P + M.off(3), M.h2);
    gemm(s, (int)b, M.nout, M.w, M.h2, M.w, 1, W3, M.w, 1, M.y, M.nout);
    bias_add<<<nblk(b * M.nout), 256, 0, s>>>(b, M.nout, M.y, M.P + M.off(5));
}

// gradient of sum((y - t)^2) / (2 n_total) over a batch, accumulated into M.G (beta = 1) or written (beta = 0)
static void mlp_backward_batch(Mlp& M, const float* T, int64_t b, double n_total, float beta, cudaStream_t s) {
    mse_grad<<<nblk(b * M.nout), 256, 0, s>>>(b * M.nout, M.y, T, (float)(1.0 / n_total), M.dyb, M.loss);
    const bf16 *W2 = M.Pb + M.off(2), *W3 = M.Pb + M.off(4);
    // dW3 [nout][w] = dy^T h2 : A(m = o, k = r) = dy[r][o], B(n = j, k = r) = h2[r][j]
    gemm(s, M.nout, M.w, (int)b, M.dyb, 1, M.nout, M.h2, 1, M.w, M.G + M.off(4), M.w, 1.f, beta);
    col_sum<<<(M.nout + 127) / 128, 128, 0, s>>>(b, M.nout, M.dyb, M.G + M.off(5), beta != 0.f);
    // dh2 [b][w] = dy W3 : A(m = r, k = o) = dy[r][o], B(n = j, k = o) = W3[o][j]
    gemm(s, (int)b, M.w, M.nout, M.dyb, M.nout, 1, W3, 1, M.w, M.dh2, M.w);
    relu_back<<<nblk(b * M.w), 256, 0, s>>>(b * M.w, M.dh2, M.z2, M.dz2);
    gemm(s, M.w, M.w, (int)b, M.dz2, 1, M.w, M.h1, 1, M.w, M.G + M.off(2), M.w, 1.f, beta);
    col_sum<<<(M.w + 127) / 128, 128, 0, s>>>(b, M.w, M.dz2, M.G + M.off(3), beta != 0.f);
    gemm(s, (int)b, M.w, M.w, M.dz2, M.w, 1, W2, 1, M.w, M.dh1, M.w);
    relu_back<<<nblk(b * M.w), 256, 0, s>>>(b * M.w, M.dh1, M.z1, M.dz1);
    gemm(s, M.w, M.nin_pad, (int)b, M.dz1, 1, M.w, M.xb, 1, M.nin_pad, M.G + M.off(0), M.nin_pad, 1.f, beta);
    col_sum<<<(M.w + 127) / 128, 128, 0, s>>>(b, M.w, M.dz1, M.G + M.off(1), beta != 0.f);
}

// forward and gradient of a batch
static void mlp_step(Mlp& M, const float* X, int64_t ldx, const float* T, int64_t b, double n_total, float beta, cudaStream_t s) {
    if (mlp_fast(M, T)) { mlp_step_fused(M, X, ldx, T, b, n_total, beta, s); return; }
    mlp_forward_batch(M, X, ldx, b, s);
    mlp_backward_batch(M, T, b, n_total, beta, s);
}

int mlp_create(int nin, int width, int nout, uint64_t seed, Mlp** out, std::string& err) {
    Mlp* M = new Mlp();
    M->nin = nin;
    M->nin_pad = (nin + 15) / 16 * 16;
    M->w = width;
    M->nout = nout;
    M->nparam = M->off(5) + nout;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&M->n_sm, cudaDevAttrMultiProcessorCount, dev);
    std::vector<float> h(M->nparam, 0.f);
    // He-uniform initial weights from SplitMix64 (biases zero)
    uint64_t st = seed * 0x9E3779B97F4A7C15ull + 1;
    auto next = [&]() {
        uint64_t z = (st += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        return ((z >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    };
    auto fill = [&](int k, int fan_in, int rows, int cols, int ld) {
        const double lim = std::sqrt(6.0 / fan_in);
        for (int r = 0; r < rows; ++r)
            for (int c = 0; c < cols; ++c) h[M->off(k) + (int64_t)r * ld + c] = (float)((2.0 * next() - 1.0) * lim);
    };
    fill(0, nin, width, nin, M->nin_pad);
    fill(2, width, width, width, width);
    fill(4, width, nout, width, width);
    for (int64_t i = M->off(4); i < M->off(5); ++i) h[i] *= 0.1f;   // small initial output
    bool ok = cudaMalloc((void**)&M->P, M->nparam * 4) == cudaSuccess && cudaMalloc((void**)&M->G, M->nparam * 4) == cudaSuccess &&
              cudaMalloc((void**)&M->Mm, M->nparam * 4) == cudaSuccess && cudaMalloc((void**)&M->Vm, M->nparam * 4) == cudaSuccess &&
              cudaMalloc((void**)&M->Pb, M->nparam * 2) == cudaSuccess && cudaMalloc((void**)&M->loss, 8) == cudaSuccess;
    if (!ok) { err = "MLP allocation failed"; delete M; return 1; }
    cudaMemcpy(M->P, h.data(), M->nparam * 4, cudaMemcpyHostToDevice);
    cudaMemset(M->G, 0, M->nparam * 4);
    cudaMemset(M->Mm, 0, M->nparam * 4);
    cudaMemset(M->Vm, 0, M->nparam * 4);
    mlp_sync_bf16(*M, 0);
    *out = M;
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}

void mlp_destroy(Mlp* M) {
    if (!M) return;
    void* p[] = {M->P, M->G, M->Mm, M->Vm, M->Pb, M->loss, M->xb, M->h1, M->h2, M->dyb, M->dz2, M->dz1, M->z1, M->z2, M->y, M->dh2, M->dh1};
    for (void* q : p) if (q) cudaFree(q);
    delete M;
}

int64_t mlp_nparam(const Mlp* M) { return M->nparam; }
int mlp_nin_pad(const Mlp* M) { return M->nin_pad; }

int mlp_params(Mlp* M, float* host, int set) {
    if (set) {
        cudaMemcpy(M->P, host, M->nparam * 4, cudaMemcpyHostToDevice);
        cudaMemset(M->Mm, 0, M->nparam * 4);
        cudaMemset(M->Vm, 0, M->nparam * 4);
        M->step = 0;
        mlp_sync_bf16(*M, 0);
    } else {
        cudaMemcpy(host, M->P, M->nparam * 4, cudaMemcpyDeviceToHost);
    }
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}

int mlp_grads(Mlp* M, float* host) { return cudaMemcpy(host, M->G, M->nparam * 4, cudaMemcpyDeviceToHost) == cudaSuccess ? 0 : 1; }

int mlp_forward(Mlp* M, const float* X, int64_t ldx, int64_t n, float* Y, cudaStream_t s) {
    const int64_t B = 4096;
    // (in place, or overlapping otherwise: batch by batch, each read whole before its results are written)
    const bool apart = (uintptr_t)(Y + n * M->nout) <= (uintptr_t)X || (uintptr_t)(X + (n - 1) * ldx + M->nin) <= (uintptr_t)Y;
    if (mlp_fast(*M, Y) && (apart || n == 0)) {
        if (n > 0) mlp_fused_rows<false>(*M, X, ldx, n, Y, MlpTrainIO{}, s);
        return cudaGetLastError() == cudaSuccess ? 0 : 1;
    }
    if (!mlp_reserve(*M, std::min(n, B), true)) return 1;
    for (int64_t r = 0; r < n; r += B) {
        const int64_t b = std::min(B, n - r);
        mlp_forward_batch(*M, X + r * ldx, ldx, b, s);
        cudaMemcpyAsync(Y + r * M->nout, M->y, b * M->nout * 4, cudaMemcpyDeviceToDevice, s);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

// gradient of the mean loss over all n samples (one pass, no update); returns the loss
int mlp_gradient(Mlp* M, const float* X, int64_t ldx, const float* T, int64_t n, double* loss, cudaStream_t s) {
    const int64_t B = 4096;
    if (!mlp_reserve(*M, std::min(n, B), !mlp_fast(*M, T))) return 1;
    cudaMemsetAsync(M->loss, 0, 8, s);
    for (int64_t r = 0; r < n; r += B) {
        const int64_t b = std::min(B, n - r);
        mlp_step(*M, X + r * ldx, ldx, T + r * M->nout, b, (double)n, r == 0 ? 0.f : 1.f, s);
    }
    double h = 0.0;
    cudaMemcpyAsync(&h, M->loss, 8, cudaMemcpyDeviceToHost, s);
    cudaStreamSynchronize(s);
    *loss = h / (2.0 * (double)n);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

// Adam over shuffled-free mini-batches; loss_hist[e] = mean training loss of epoch e
int mlp_train(Mlp* M, const float* X, int64_t ldx, const float* T, int64_t n, int epochs, int batch, float lr,
              double* loss_hist, cudaStream_t s) {
    if (!mlp_reserve(*M, std::min<int64_t>(n, batch), !mlp_fast(*M, T))) return 1;
    for (int ep = 0; ep < epochs; ++ep) {
        cudaMemsetAsync(M->loss, 0, 8, s);
        for (int64_t r = 0; r < n; r += batch) {
            const int64_t b = std::min<int64_t>(batch, n - r);
            mlp_step(*M, X + r * ldx, ldx, T + r * M->nout, b, (double)b, 0.f, s);
            ++M->step;
            const float b1 = 0.9f, b2 = 0.999f;
            const float c1 = 1.f / (1.f - std::pow(b1, (float)M->step)), c2 = 1.f / (1.f - std::pow(b2, (float)M->step));
            adam<<<nblk(M->nparam), 256, 0, s>>>(M->nparam, M->P, M->G, M->Mm, M->Vm, M->Pb, lr, b1, b2, 1e-8f, c1, c2);
        }
        double h = 0.0;
        cudaMemcpyAsync(&h, M->loss, 8, cudaMemcpyDeviceToHost, s);
        cudaStreamSynchronize(s);
        if (loss_hist) loss_hist[ep] = h / (2.0 * (double)n);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

// ------------------------------------------------------------------------------------------
// preconditioner data: features, targets, corrections
// ------------------------------------------------------------------------------------------
int precond_dataset(const Mesh& m, const double* u, const double* up, const double* up2, const double* f,
                    const imga_physics& ph, int precision, const int32_t* elems, int64_t n, int ldx, float* X,
                    float* T, float* scale, double* Kbuf, cudaStream_t s) {
    if (n <= 0) return 0;
    if (element_jacobians(m, u, up, up2, f, ph, precision, elems, n, Kbuf, s)) return 1;
    Args A = make_args(m, u, up, up2, f, ph, nullptr, nullptr);
    dataset_kernel<<<(unsigned)((n * 32 + 127) / 128), 128, 0, s>>>(A, n, elems, Kbuf, m.d.marker, kTargetShift, ldx, X, T, scale);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int precond_correction(const Mesh& m, const imga_physics& ph, const int32_t* elems, int64_t n, const float* C,
                       const float* scale, float omega, const double* v, double* zc, double* z, cudaStream_t s) {
    const int64_t nn = m.n_nodes();
    cudaMemsetAsync(zc, 0, nn * 4 * sizeof(double), s);
    Args A = make_args(m, v, v, v, nullptr, ph, nullptr, zc);
    if (n > 0) correction_apply<<<(unsigned)((n * 32 + 127) / 128), 128, 0, s>>>(A, n, elems, C, scale, omega, v, zc);
    if (nn > 0)
        combine_rows<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(nn, m.d.bcflag, m.user_bc ? m.d.bcmask_user : nullptr, zc, z);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int gemm_bf16_test(int M, int N, int K, const float* A, const float* B, float* C, cudaStream_t s) {
    bf16 *a = nullptr, *b = nullptr;
    if (cudaMalloc((void**)&a, (size_t)M * K * 2) != cudaSuccess || cudaMalloc((void**)&b, (size_t)N * K * 2) != cudaSuccess) return 1;
    to_bf16<<<nblk((int64_t)M * K), 256, 0, s>>>((int64_t)M * K, A, a);
    to_bf16<<<nblk((int64_t)N * K), 256, 0, s>>>((int64_t)N * K, B, b);
    gemm(s, M, N, K, a, K, 1, b, K, 1, C, N);
    cudaStreamSynchronize(s);
    cudaFree(a);
    cudaFree(b);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

}  // namespace imga
