// Level-2 preconditioner of Algorithm 1, step 4, on sm_103a:
//   M2 = C~^T C~ + lambda~ W   (s x s, assembled in FP64),
//   M2 + nu I = L L^T          (FP64 Cholesky; nu = 0, then the stabilising
//                               shift retries described in msp.h),
//   L^{-1}                     (FP64), stored in the working precision as
//                               B = L^{-1} and B^T so that the level-2
//                               iteration applies M2^{-1} v = B^T (B v).
// FP32 sketches: the factor and its inverse in float-float, by block elimination on 32 x
// 32 tiles in one launch (k_chol_inv_ff). FP64 ones: a recursion that halves the matrix,
//   [A11 . ; A21 A22]:  (L11, X11) = f(A11);  L21 = A21 X11^T;
//   A22 -= L21 L21^T;   (L22, X22) = f(A22);  X21 = -X22 (L21 X11),
// with a one-block Cholesky + inverse at the leaves (at most 32 x 32) and an
// FP64 GEMM kernel for the rest; L21 X11 runs on a side stream beside the
// factorisation of A22.
#include "bulk.cuh"
#include "msp_internal.cuh"

#include <atomic>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

namespace {

// ----------------------------------------------------------- Gram (SIMT)

// M2[a][b] = sum_k Ct[k][a] Ct[k][b] + lam_t * W[a][b], FP64 output; pad rows
// (a >= s or b >= s) get the identity. One 64 x 64 tile of the upper
// triangle per block (mirrored), 256 threads each 4 x 4 outputs, K chunks of
// 16 from shared memory. Each chunk is summed in TA, then added into an
// (hi, lo) pair with Knuth's TwoSum (compensated summation), so the
// accumulated rounding error does not grow with K (K = n when Phi = I).
template <typename TA>
__device__ inline void two_sum_add(TA& hi, TA& lo, TA v) {
    TA s = hi + v;
    TA bp = s - hi;
    TA err = (hi - (s - bp)) + (v - bp);
    hi = s;
    lo += err;
}

// Split-K slices of the Gram (combined in FP64): at least 4, and as many as give
// each SM about a block, 64 rows or more a slice, up to 32. The Grams of the sketch
// sizes below 512 have 1 to 10 tiles: with 4 slices whatever the size, that of 4999 x
// 384 (FP32) took 208 us on 24 blocks and that of 1024 x 128 in FP64 425 us on
// 12; they take 66 and 110 us.
constexpr int kGramSlicesMax = 32;
constexpr int kGemmSlices = 4;   // split-K slices of k_gemm_tn

int gram_slices(const msp_ctx* ctx, int64_t tiles, int64_t K) {
    const int64_t want = std::min<int64_t>(kGramSlicesMax, std::min<int64_t>(ctx->num_sms / tiles, K / 64));
    return (int)std::max<int64_t>(4, want);
}

// Partial Gram of one K slice: P[slice][a][b] = sum_{k in slice} Ct[k][a] Ct[k][b]
// for the upper-triangular 64 x 64 tile pairs (mirrored) of the first nt tiles a side,
// FP64 output (hi + lo). blockIdx.x = tile pair, blockIdx.y = K slice.
template <typename TA>
__global__ void __launch_bounds__(256, 4) k_gram(const TA* __restrict__ Ct, int64_t K, int64_t ld,
                                                int64_t s_pad, int nt, double* __restrict__ P) {
    __shared__ __align__(16) TA As[16][64];
    __shared__ __align__(16) TA Bs[16][64];
    int ta = 0, rem = blockIdx.x;
    while (rem >= nt - ta) { rem -= nt - ta; ++ta; }
    const int tb = ta + rem;
    const int a0 = ta * 64, b0 = tb * 64;
    const int64_t kper = ((K + gridDim.y - 1) / gridDim.y + 15) / 16 * 16;
    const int64_t kbeg = (int64_t)blockIdx.y * kper;
    const int64_t kend = min(K, kbeg + kper);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    TA hi[4][4], lo[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { hi[i][j] = TA(0); lo[i][j] = TA(0); }
    for (int64_t k0 = kbeg; k0 < kend; k0 += 16) {
        for (int e = threadIdx.x; e < 16 * 64; e += 256) {
            int kk = e >> 6, cc = e & 63;
            bool in = (k0 + kk) < kend;
            As[kk][cc] = in ? Ct[(k0 + kk) * ld + a0 + cc] : TA(0);
            Bs[kk][cc] = in ? Ct[(k0 + kk) * ld + b0 + cc] : TA(0);
        }
        __syncthreads();
        TA acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = TA(0);
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            TA av[4], bv[4];
            if constexpr (sizeof(TA) == 4) {
                const float4 va = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
                const float4 vb = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
                av[0] = va.x; av[1] = va.y; av[2] = va.z; av[3] = va.w;
                bv[0] = vb.x; bv[1] = vb.y; bv[2] = vb.z; bv[3] = vb.w;
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) av[i] = As[kk][ty * 4 + i];
#pragma unroll
                for (int j = 0; j < 4; ++j) bv[j] = Bs[kk][tx * 4 + j];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) two_sum_add(hi[i][j], lo[i][j], acc[i][j]);
        __syncthreads();
    }
    double* Ps = P + (int64_t)blockIdx.y * s_pad * s_pad;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t a = a0 + ty * 4 + i, b = b0 + tx * 4 + j;
            const double v = (double)hi[i][j] + (double)lo[i][j];
            Ps[a * s_pad + b] = v;
            Ps[b * s_pad + a] = v;
        }
}

// M2 = sum_slices P + lam_t W (FP64, fixed order), or + lam_t I when W is
// NULL; pad rows/cols get identity.
// The same partial Grams (FP32 input) with 128 x 128 tiles: 512 threads,
// each 8 rows (ty*4 + i and 64 + ty*4 + i) x 4 columns (tx*4 + j), K chunks
// of 16 double-buffered in shared memory by 16-byte async copies. Per output
// the arithmetic is k_gram's -- chunks of 16 summed in FP32 from zero in
// increasing k, TwoSum into (hi, lo) -- so P is the same to the bit for the same K slices
// (their number follows the tiles, so it can differ); a thread's 32 outputs per shared-memory read of 12 values (4
// for k_gram's 16) keep the FP32 pipe, not shared memory, the limit.
__global__ void __launch_bounds__(512, 1) k_gram128(const float* __restrict__ Ct, int64_t K, int64_t ld,
                                                    int64_t s_pad, int nt, double* __restrict__ P) {
    __shared__ __align__(16) float As[2][16][128];
    __shared__ __align__(16) float Bs[2][16][128];
    int ta = 0, rem = blockIdx.x;
    while (rem >= nt - ta) { rem -= nt - ta; ++ta; }
    const int tb = ta + rem;
    const int a0 = ta * 128, b0 = tb * 128;
    const int64_t kper = ((K + gridDim.y - 1) / gridDim.y + 15) / 16 * 16;
    const int64_t kbeg = (int64_t)blockIdx.y * kper;
    const int64_t kend = min(K, kbeg + kper);
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    // loader: thread t copies float4 (t & 31) of row t >> 5 of the chunk, of A and of B
    const int lk = (int)(threadIdx.x >> 5), lc = (int)(threadIdx.x & 31) * 4;
    auto issue = [&](int64_t k0, int st) {
        const int64_t k = k0 + lk;
        const bool in = k < kend;
        msp::cp_async16(&As[st][lk][lc], in ? Ct + k * ld + a0 + lc : Ct, in);
        msp::cp_async16(&Bs[st][lk][lc], in ? Ct + k * ld + b0 + lc : Ct, in);
    };
    float hi[8][4], lo[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { hi[i][j] = 0.f; lo[i][j] = 0.f; }
    if (kbeg < kend) issue(kbeg, 0);
    msp::cp_async_commit();
    int st = 0;
    for (int64_t k0 = kbeg; k0 < kend; k0 += 16) {
        if (k0 + 16 < kend) issue(k0 + 16, st ^ 1);
        msp::cp_async_commit();
        msp::cp_async_wait<1>();
        __syncthreads();
        float acc[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            const float4 x0 = *reinterpret_cast<const float4*>(&As[st][kk][ty * 4]);
            const float4 x1 = *reinterpret_cast<const float4*>(&As[st][kk][64 + ty * 4]);
            const float4 y = *reinterpret_cast<const float4*>(&Bs[st][kk][tx * 4]);
            const float av[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
            const float bv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) two_sum_add(hi[i][j], lo[i][j], acc[i][j]);
        __syncthreads();
        st ^= 1;
    }
    double* Ps = P + (int64_t)blockIdx.y * s_pad * s_pad;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t a = a0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + (i - 4)), b = b0 + tx * 4 + j;
            const double v = (double)hi[i][j] + (double)lo[i][j];
            Ps[a * s_pad + b] = v;
            Ps[b * s_pad + a] = v;
        }
}

// Split-K partial Grams of the first s columns of Ct into scratch P (*slices x s_pad x
// s_pad, with `extra` doubles behind them).
template <typename TA>
msp_status launch_gram(msp_ctx* ctx, const TA* Ct, int64_t K, int64_t ld, int64_t s, int64_t sp, int64_t extra,
                       double** P, int* slices) {
    const bool wide = sizeof(TA) == 4 && sp % 128 == 0 && ld % 4 == 0 && ((uintptr_t)Ct & 15) == 0;
    const int nt = (int)((s + (wide ? 127 : 63)) / (wide ? 128 : 64));     // tiles of padding are not read
    const int tiles = nt * (nt + 1) / 2;
    *slices = gram_slices(ctx, tiles, K);
    void* scr = nullptr;
    MSP_TRY(msp_scratch(ctx, (size_t)(*slices * sp * sp + extra) * 8, &scr));
    *P = (double*)scr;
    const dim3 grid((unsigned)tiles, (unsigned)*slices);
    if constexpr (sizeof(TA) == 4) {
        if (wide) {
            k_gram128<<<grid, 512, 0, ctx->stream>>>(Ct, K, ld, sp, nt, *P);
            MSP_CHECK_LAUNCH(ctx);
            return MSP_OK;
        }
    }
    k_gram<TA><<<grid, 256, 0, ctx->stream>>>(Ct, K, ld, sp, nt, *P);
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

template <typename TA>
__global__ void k_gram_finish(const double* __restrict__ P, int slices, const TA* __restrict__ W, double lam_t,
                              int64_t s, int64_t s_pad, double* __restrict__ M2) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= s_pad * s_pad) return;
    const int64_t a = e / s_pad, b = e % s_pad;
    double v;
    if (a < s && b < s) {
        v = 0.0;
#pragma unroll 4
        for (int sl = 0; sl < slices; ++sl) v += P[(int64_t)sl * s_pad * s_pad + e];
        v += W ? lam_t * (double)W[e] : (a == b ? lam_t : 0.0);
    } else {
        v = (a == b) ? 1.0 : 0.0;
    }
    M2[e] = v;
}

// W <- (W + W^T)/2 in place (working precision) and W64 = (double)W.
template <typename T>
__global__ void k_symmetrize(T* __restrict__ W, double* __restrict__ W64, int64_t s_pad) {
    int64_t a = blockIdx.y * 32 + threadIdx.y, b = blockIdx.x * 32 + threadIdx.x;
    if (a >= s_pad || b >= s_pad || b > a) return;
    T v = (W[a * s_pad + b] + W[b * s_pad + a]) * T(0.5);
    W[a * s_pad + b] = v;
    W[b * s_pad + a] = v;
    W64[a * s_pad + b] = (double)v;
    W64[b * s_pad + a] = (double)v;
}

// ----------------------------------------------------------- FP64 GEMM

// Cm = alpha * op(A) op(B) + beta * Cm, row-major; op(A) is m x k, op(B) k x n.
// TS x TS output tile (TS = 16 or 32), 256 threads, K chunks of 16. The
// triangular structure of the operands limits the K range of each tile:
//   tri_a = 1: op(A) lower triangular (A[i][k] = 0 for k > i)
//   tri_b = 1: op(B) upper triangular (B[k][j] = 0 for k > j)
//   tri_b = 2: op(B) lower triangular (B[k][j] = 0 for k < j)
//   lower_out: only tiles touching the lower triangle (i >= j) are computed.
template <bool TA_, bool TB_, int TS>
__global__ void __launch_bounds__(256) k_dgemm(int64_t m, int64_t n, int64_t k, double alpha,
                                              const double* __restrict__ A, int64_t lda,
                                              const double* __restrict__ B, int64_t ldb,
                                              double beta, double* __restrict__ Cm, int64_t ldc,
                                              int tri_a, int tri_b, int lower_out) {
    constexpr int PT = TS / 16;              // outputs per thread per dimension
    __shared__ double As[16][TS + 1];        // As[kk][i] = op(A)[i][k0+kk]
    __shared__ double Bs[16][TS + 1];        // Bs[kk][j] = op(B)[k0+kk][j]
    const int64_t i0 = (int64_t)blockIdx.y * TS, j0 = (int64_t)blockIdx.x * TS;
    if (lower_out && j0 > i0 + TS - 1) return;
    int64_t kbeg = 0, kend = k;
    if (tri_a == 1) kend = min(kend, i0 + TS);
    if (tri_b == 1) kend = min(kend, j0 + TS);
    if (tri_b == 2) kbeg = (j0 / 16) * 16;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double acc[PT][PT];
#pragma unroll
    for (int i = 0; i < PT; ++i)
#pragma unroll
        for (int j = 0; j < PT; ++j) acc[i][j] = 0.0;
    for (int64_t k0 = kbeg; k0 < kend; k0 += 16) {
        for (int e = threadIdx.x; e < 16 * TS; e += 256) {
            int kk, ii;
            if (TA_) { ii = e % TS; kk = e / TS; }   // A^T: read A[k][i], contiguous in i
            else { kk = e & 15; ii = e >> 4; }        // A: read A[i][k], contiguous in k
            int64_t gi = i0 + ii, gk = k0 + kk;
            double v = 0.0;
            if (gi < m && gk < kend) v = TA_ ? A[gk * lda + gi] : A[gi * lda + gk];
            As[kk][ii] = v;
        }
        for (int e = threadIdx.x; e < 16 * TS; e += 256) {
            int kk, jj;
            if (TB_) { kk = e & 15; jj = e >> 4; }    // B^T: read B[j][k], contiguous in k
            else { jj = e % TS; kk = e / TS; }        // B: read B[k][j], contiguous in j
            int64_t gj = j0 + jj, gk = k0 + kk;
            double v = 0.0;
            if (gj < n && gk < kend) v = TB_ ? B[gj * ldb + gk] : B[gk * ldb + gj];
            Bs[kk][jj] = v;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            double av[PT], bv[PT];
#pragma unroll
            for (int i = 0; i < PT; ++i) av[i] = As[kk][ty * PT + i];
#pragma unroll
            for (int j = 0; j < PT; ++j) bv[j] = Bs[kk][tx * PT + j];
#pragma unroll
            for (int i = 0; i < PT; ++i)
#pragma unroll
                for (int j = 0; j < PT; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < PT; ++i)
#pragma unroll
        for (int j = 0; j < PT; ++j) {
            int64_t gi = i0 + ty * PT + i, gj = j0 + tx * PT + j;
            if (gi < m && gj < n) {
                double c = beta == 0.0 ? 0.0 : beta * Cm[gi * ldc + gj];
                Cm[gi * ldc + gj] = c + alpha * acc[i][j];
            }
        }
}

// ----------------------------------------------------- float-float kernels
//
// The factor of an FP32 sketch runs in float-float arithmetic on the FP32
// pipe: a value is the unevaluated sum hi + lo of two floats (|lo| <= ulp(hi)
// / 2 once normalised), a product is exact by FMA (TwoProduct, Dekker), a sum
// by TwoSum (Knuth), about 2^-46 relative per operation. FP64 runs at 2
// lanes per clock per SM on this part, the FP32 pipe at 128. Every operation
// below uses the _rn intrinsics, which the compiler never contracts.

__device__ __forceinline__ float2 ff_fast2sum(float a, float b) {   // needs |a| >= |b| or a = 0
    const float s = __fadd_rn(a, b);
    return make_float2(s, __fsub_rn(b, __fsub_rn(s, a)));
}

__device__ __forceinline__ float2 ff_2sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}

// (sh, sl) += a b, sl collecting the low parts until the next ff_norm
__device__ __forceinline__ void ff_fma_acc(float& sh, float& sl, float2 a, float2 b) {
    const float p = __fmul_rn(a.x, b.x);
    float e = __fmaf_rn(a.x, b.x, -p);
    e = __fmaf_rn(a.x, b.y, e);
    e = __fmaf_rn(a.y, b.x, e);
    const float2 t = ff_2sum(sh, p);
    sh = t.x;
    sl = __fadd_rn(sl, __fadd_rn(t.y, e));
}

__device__ __forceinline__ float2 ff_norm(float sh, float sl) { return ff_2sum(sh, sl); }

__device__ __forceinline__ float2 ff_mul(float2 a, float2 b) {
    const float p = __fmul_rn(a.x, b.x);
    float e = __fmaf_rn(a.x, b.x, -p);
    e = __fmaf_rn(a.x, b.y, e);
    e = __fmaf_rn(a.y, b.x, e);
    return ff_fast2sum(p, e);
}

__device__ __forceinline__ float2 ff_add(float2 a, float2 b) {
    const float2 s = ff_2sum(a.x, b.x);
    return ff_fast2sum(s.x, __fadd_rn(s.y, __fadd_rn(a.y, b.y)));
}

__device__ __forceinline__ float2 ff_from_double(double v) {
    const float h = __double2float_rn(v);
    return make_float2(h, __double2float_rn(v - (double)h));
}

__device__ __forceinline__ double ff_to_double(float2 a) { return (double)a.x + (double)a.y; }

constexpr int kLeafSmem = 2 * 64 * 65 * (int)sizeof(double);
constexpr int kLeafUpd = 256;                 // eight update warps (32 x 8 thread grid)
constexpr int kLeafThreads = kLeafUpd + 32;   // and the pivot warp

// 1/sqrt(d) for a positive normal FP64 d: FP32 reciprocal square root as the
// seed, then two Newton-Raphson steps y <- y (3 - d y^2) / 2 for f(y) =
// 1/y^2 - d (quadratic convergence: ~2^-22 -> 2^-44 -> FP64 rounding). The
// FP64 square root and division cost tens of FP64 instructions each on this
// part, whose FP64 unit takes ~64 cycles per warp instruction.
__device__ inline double rsqrt_newton(double d) {
    if (!(d >= 1e-30 && d <= 1e30)) return 1.0 / sqrt(d);
    double y = (double)rsqrtf((float)d);
    const double hd = 0.5 * d;
    y = y * fma(-hd * y, y, 1.5);
    y = y * fma(-hd * y, y, 1.5);
    return y;
}

// 1/d for a positive normal FP64 d: FP32 reciprocal as the seed, then two
// Newton-Raphson steps r <- r + r (1 - d r) for f(r) = 1/r - d.
__device__ inline double rcp_newton(double d) {
    if (!(d >= 1e-30 && d <= 1e30)) return 1.0 / d;
    double r = (double)(1.0f / (float)d);
    r = fma(r, fma(-d, r, 1.0), r);
    r = fma(r, fma(-d, r, 1.0), r);
    return r;
}

// Cholesky and inverse of an nb x nb (nb <= 64; the recursion passes at most
// 32) FP64 block on one SM:
// M = L L^T (lower triangle of M overwritten with L), X = L^{-1}.
// One elimination sweep in LDL^T form: at step k every row i > k takes
// t_i = a_ik / d_k and updates both its Schur-complement entries,
// a_ij -= t_i a_jk (k < j < i), and its row of X, x_ij -= t_i x_kj (j <= k),
// with X starting as the identity -- the same row operations turn the
// identity into L_u^{-1} for A = L_u D L_u^T. Every update of a step is
// independent (no substitution chains), and the two parts together keep the
// work per step near n^2 / 2. The diagonal is kept apart by a fifth warp,
// which also forms the next pivot d_{k+1} and 1/d_{k+1} while the update
// warps work, so a step costs one barrier. At the end L = L_u D^{1/2}
// (l_ik = a_ik / sqrt(d_k), l_kk = sqrt(d_k)) and L^{-1} = D^{-1/2} L_u^{-1}.
// A pivot that is not positive and finite sets *fail (and is replaced by 1).
__global__ void __launch_bounds__(kLeafThreads) k_chol_leaf(double* __restrict__ M, double* __restrict__ X,
                                                           int64_t ld, int nb, int* __restrict__ fail) {
    extern __shared__ __align__(16) double leaf_smem[];
    double (*a)[65] = reinterpret_cast<double (*)[65]>(leaf_smem);
    double (*x)[65] = reinterpret_cast<double (*)[65]>(leaf_smem + 64 * 65);
    __shared__ double piv[64], rinv[64], rs[64];
    __shared__ int bad;
    const int tid = threadIdx.x, lane = tid & 31;
    const bool pivot_warp = tid >= kLeafUpd;
    if (tid == 0) bad = 0;
    for (int e = tid; e < nb * nb; e += kLeafThreads) {
        const int i = e / nb, j = e % nb;
        a[i][j] = (j <= i) ? M[i * ld + j] : 0.0;
        x[i][j] = (i == j) ? 1.0 : 0.0;
    }
    __syncthreads();
    // pivot warp: the diagonal of rows lane and lane + 32
    double dg0 = 1.0, dg1 = 1.0;
    if (pivot_warp) {
        if (lane < nb) dg0 = a[lane][lane];
        if (lane + 32 < nb) dg1 = a[lane + 32][lane + 32];
        if (lane == 0) {
            double d = dg0;
            if (!(d > 0.0) || !isfinite(d)) {
                bad = 1;
                d = 1.0;
            }
            piv[0] = d;
            rinv[0] = rcp_newton(d);
        }
    }
    __syncthreads();
    // update threads: row offsets interleaved over the warps, so that the
    // last steps (few rows) still use all eight
    const int tx = tid & 7, ty = tid >> 3;
    const int rr = ((ty & 3) << 3) | (ty >> 2);
    for (int k = 0; k < nb; ++k) {
        const double rk = rinv[k];
        if (!pivot_warp) {
            for (int i = k + 1 + rr; i < nb; i += 32) {
                const double ti = a[i][k] * rk;
                for (int j = tx; j <= k; j += 8) x[i][j] = fma(-ti, x[k][j], x[i][j]);
                for (int j = k + 1 + tx; j < i; j += 8) a[i][j] = fma(-ti, a[j][k], a[i][j]);
            }
        } else if (k + 1 < nb) {
            if (lane > k && lane < nb) {
                const double ti = a[lane][k] * rk;
                dg0 = fma(-ti, a[lane][k], dg0);
            }
            if (lane + 32 > k && lane + 32 < nb) {
                const double ti = a[lane + 32][k] * rk;
                dg1 = fma(-ti, a[lane + 32][k], dg1);
            }
            const int kn = k + 1;
            if (lane == (kn & 31)) {
                double d = kn < 32 ? dg0 : dg1;
                if (!(d > 0.0) || !isfinite(d)) {
                    bad = 1;
                    d = 1.0;
                }
                piv[kn] = d;
                rinv[kn] = rcp_newton(d);
            }
        }
        __syncthreads();
    }
    for (int k = tid; k < nb; k += kLeafThreads) rs[k] = rsqrt_newton(piv[k]);
    __syncthreads();
    for (int e = tid; e < nb * nb; e += kLeafThreads) {
        const int i = e / nb, j = e % nb;
        if (j < i) M[i * ld + j] = a[i][j] * rs[j];
        else if (j == i) M[i * ld + j] = piv[i] * rs[i];
        X[i * ld + j] = (j <= i) ? x[i][j] * rs[i] : 0.0;
    }
    if (tid == 0 && bad) atomicExch(fail, 1);
}

// d^{-1/2} in float-float for a positive normal d: the FP32 rsqrtf r0, then
// one Newton-Raphson step r = r0 + r0 (1 - d r0^2) / 2 with the residual
// 1 - d r0^2 formed to first order exactly (r0^2 and d r0^2 by TwoProduct;
// d r0^2 is within about 2^-21 of 1), ~2^-43 relative.
__device__ __forceinline__ float2 ff_rsqrt(float2 d) {
    const float r0 = rsqrtf(d.x);
    const float th = __fmul_rn(r0, r0), tl = __fmaf_rn(r0, r0, -th);
    const float p = __fmul_rn(d.x, th);
    const float pe = __fmaf_rn(d.y, th, __fmaf_rn(d.x, tl, __fmaf_rn(d.x, th, -p)));
    const float res = __fsub_rn(__fsub_rn(1.0f, p), pe);
    return ff_fast2sum(r0, __fmul_rn(__fmul_rn(0.5f, r0), res));
}

// Element (i, j) of a float-float matrix kept as 32 x 32 row-major tiles.
__device__ __forceinline__ int64_t ff_tile_at(int64_t i, int64_t j, int64_t s_pad) {
    return (((i >> 5) * (s_pad >> 5) + (j >> 5)) << 10) + ((i & 31) << 5) + (j & 31);
}

constexpr int kFFThreads = 288;     // eight warps of the tiles, and the leaf's pivot warp

struct FFShared {
    float4 L[512], R[512];            // a tile's operands, k-major: [k][row or column]
    float2 T[32][33];                 // the leaf, or the pivot tile's inverse
    float2 A[32][33];                 // block 0: the tile below the pivot
    float2 row[2][32], rk[2], piv[32];
    int bad;
};

// 1/d in float-float for a positive normal d: r0, the hardware's approximation
// (2^-23 relative), then a Newton-Raphson step for f(r) = 1/r - d carried to second order,
// r = r0 + r0 (e + e^2), with the residual e = 1 - d r0 formed to
// first order exactly (1 - hi(d r0) is exact), ~2^-46 relative. The low part may
// overlap the high one by a bit or two. (|X M X^T - I| of the whole factor against the one
// before, which started from a rounded reciprocal and normalised every product: 1.04 times
// at s_pad = 128 with s = 60, 0.76 at 128, 0.47, 0.27 and 0.16 at 256, 512 and 1024.)
__device__ __forceinline__ float2 ff_rcp(float2 d) {
    float r0;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(d.x));
    const float p = __fmul_rn(d.x, r0);
    const float pe = __fmaf_rn(d.y, r0, __fmaf_rn(d.x, r0, -p));
    const float res = __fsub_rn(__fsub_rn(1.0f, p), pe);
    return make_float2(r0, __fmul_rn(r0, __fmaf_rn(res, res, res)));
}

// -a b, the parts not renormalised (what ff_fma_acc takes as well)
__device__ __forceinline__ float2 ff_nmul(float2 a, float2 b) {
    const float p = __fmul_rn(a.x, -b.x);
    float e = __fmaf_rn(a.x, -b.x, -p);
    e = __fmaf_rn(a.x, -b.y, e);
    e = __fmaf_rn(a.y, -b.x, e);
    return make_float2(p, e);
}

// Cholesky inverse of the 32 x 32 tile in sh.T (both triangles), left there: the
// elimination of k_chol_leaf (LDL^T on the tile and the identity at once) in place,
// X in the columns that are done and A in the others. A lane has a column, warp w
// the rows w + 8 r in registers. Row k then is what step k adds to the rows below
// it, a_ki = a_ik times -1 / d_k the factor of row i, so a step reads the row and 1 / d_k
// from shared memory and its updates are independent of each other. A ninth warp
// keeps the diagonal and forms the next 1 / d: that chain (a product, an update, a
// reciprocal, a barrier) is what a step takes, so its products stay unnormalised
// and the test of the pivot is beside the reciprocal.
__device__ __forceinline__ void ff_leaf(FFShared& sh) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float2 zero = make_float2(0.f, 0.f), one = make_float2(1.f, 0.f);
    const bool pivots = w == 8;
    float2 v[4], dg = sh.T[lane][lane];
    auto pivot = [&](int k) {
        const float2 r = ff_rcp(dg);
        if (lane == k) {
            const bool ok = dg.x > 0.f && isfinite(dg.x);
            sh.rk[k & 1] = ok ? r : one;
            sh.piv[k] = ok ? dg : one;
            if (!ok) sh.bad = 1;
        }
    };
    if (pivots) {
        pivot(0);
    } else {
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = sh.T[w + 8 * r][lane];
        if (w == 0) sh.row[0][lane] = lane == 0 ? one : v[0];
    }
    __syncthreads();
#pragma unroll
    for (int kb = 0; kb < 4; ++kb) {
#pragma unroll 1
        for (int kr = 0; kr < (kb < 3 ? 8 : 7); ++kr) {
            const int k = 8 * kb + kr;
            const float2* row = sh.row[k & 1];
            const float2 src = row[lane], rk = sh.rk[k & 1];
            if (pivots) {
                const float2 nti = ff_nmul(src, rk);
                float h = dg.x, l = dg.y;
                ff_fma_acc(h, l, nti, src);
                dg = ff_norm(h, l);
                pivot(k + 1);
            } else {
#pragma unroll
                for (int r = kb; r < 4; ++r) {
                    const float2 nti = ff_nmul(row[w + 8 * r], rk);
                    float h = v[r].x, l = v[r].y;
                    ff_fma_acc(h, l, nti, src);
                    const float2 u = lane == k ? nti : ff_norm(h, l);
                    if (r > kb || w > kr) v[r] = u;
                }
                const float2 next = kr < 7 ? v[kb] : v[kb < 3 ? kb + 1 : 3];
                if (w == ((k + 1) & 7)) sh.row[(k + 1) & 1][lane] = lane == k + 1 ? one : next;
            }
            __syncthreads();
        }
    }
    if (!pivots) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = w + 8 * r;
            const float2 rs = ff_rsqrt(sh.piv[i]);
            sh.T[i][lane] = lane < i ? ff_mul(v[r], rs) : lane == i ? rs : zero;
        }
    }
    __syncthreads();
}

// Monotonic counters between the blocks of a cooperative launch: arrive adds one after
// the block's writes (and reads), wait_for returns once the count has reached
// `target` (false: the wait limit ran out, MSP_ETIMEOUT in *err).
__device__ __forceinline__ void arrive(unsigned int* count) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    }
}

__device__ __forceinline__ bool reached(const unsigned int* count, unsigned int target, int* err) {
    const uint64_t t0 = msp::globaltimer_ns();
    const unsigned long long limit = msp::grid_wait_limit_ns();
    while (true) {
        unsigned int cur;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(cur) : "l"(count) : "memory");
        if (cur >= target) return true;
        if (msp::globaltimer_ns() - t0 > limit) {
            atomicExch(err, (int)MSP_ETIMEOUT);
            return false;
        }
    }
}

__device__ __forceinline__ bool wait_for(const unsigned int* a, unsigned int target_a, const unsigned int* b,
                                         unsigned int target_b, int* err) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) ok = reached(a, target_a, err) && reached(b, target_b, err);
    __syncthreads();
    return ok != 0;
}

// L^{-1} of the Cholesky factor of an SPD float-float matrix of nt x nt tiles
// (tile-major, S; both triangles of the diagonal tiles), left in S's lower
// tiles: block Gauss-Jordan elimination on the matrix and the identity at once, in
// place, as tile column k is done with A before X needs it. Step k has X_kk, the
// inverse of the factor of tile (k, k), and
//   1. forms the panel L_ik = A_ik X_kk^T (i > k) into Lp, transposed, and row k of X,
//      X_kj = X_kk X_kj (j < k): a quarter of a tile a block;
//   2. updates every tile of the rows below, A_ij -= L_ik L_jk^T (j > k) and
//      X_ij -= L_ik X_kj (j <= k), a tile a block, 2 x 2 entries a thread.
// Block 0 runs one step ahead of the others: it forms L_k+1,k for itself, updates
// tile (k + 1, k + 1) and inverts its factor (ff_leaf), the next step's pivot, while they
// take the rest of step k, so that a step takes the longer of the two.
// What bounds it: block 0's chain (a leaf of about 15 thousand cycles, half of
// a step) up to s_pad = 512, the updates (14 FP32 operations a product, s_pad^3 / 3 of
// them, 135 us at s_pad = 1024 over all SMs) and the two waits beside it above. At
// s_pad = 128, 256, 512 and 1024: 55, 106, 213 and 438 us (with block 0 in step with the
// others, two grid barriers a step: 61, 121, 241 and 489 us; the recursion it
// replaced, 32 leaves and 90 dependent products at 1024: about 1200 us).
// sync (zero at the launch): failure word, -, error word, pivots published, panel
// arrivals (all blocks), update arrivals (all but block 0).
__global__ void __launch_bounds__(kFFThreads, 1) k_chol_inv_ff(float2* S, float2* Lp, int nt, int* sync) {
    __shared__ __align__(16) FFShared sh;
    const int tid = threadIdx.x, G = (int)gridDim.x, b = (int)blockIdx.x, NW = G - 1;
    const int tx = tid & 15, ty = tid >> 4, lo = tid & 7, hi = tid >> 3;
    const bool on = tid < 256;
    int* err = sync + 2;
    unsigned int* pivots = reinterpret_cast<unsigned int*>(sync + 3);
    unsigned int *panels = pivots + 1, *updates = pivots + 2;
    auto tile = [&](int i, int j) { return S + (((int64_t)i * nt + j) << 10); };
    auto load4 = [](const float2* p, int e) { return __ldcg(reinterpret_cast<const float4*>(p) + e); };
    auto stage = [&](float2 (*dst)[33], const float2* p) {
#pragma unroll
        for (int u = 0; u < 2 && on; ++u) {
            const float4 f = load4(p, 2 * tid + u);
            dst[hi][4 * lo + 2 * u] = make_float2(f.x, f.y);
            dst[hi][4 * lo + 2 * u + 1] = make_float2(f.z, f.w);
        }
    };
    // d -= Ls Rs (k-major): rows 2 ty, + 1, columns 2 tx, + 1
    auto update = [&](const float4* Ls, const float4* Rs, float4* d) {
        float s[4] = {}, e[4] = {};
#pragma unroll
        for (int k0 = 0; k0 < 2; ++k0) {
#pragma unroll 8
            for (int kk = 16 * k0; kk < 16 * k0 + 16; ++kk) {
                const float4 a = Ls[kk * 16 + ty], c = Rs[kk * 16 + tx];
                const float2 a0 = make_float2(a.x, a.y), a1 = make_float2(a.z, a.w);
                const float2 c0 = make_float2(c.x, c.y), c1 = make_float2(c.z, c.w);
                ff_fma_acc(s[0], e[0], a0, c0);
                ff_fma_acc(s[1], e[1], a0, c1);
                ff_fma_acc(s[2], e[2], a1, c0);
                ff_fma_acc(s[3], e[3], a1, c1);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float2 n = ff_norm(s[u], e[u]);
                s[u] = n.x;
                e[u] = n.y;
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float2 x = ff_add(make_float2(d[u].x, d[u].y), make_float2(-s[2 * u], -e[2 * u]));
            const float2 y = ff_add(make_float2(d[u].z, d[u].w), make_float2(-s[2 * u + 1], -e[2 * u + 1]));
            d[u] = make_float4(x.x, x.y, y.x, y.y);
        }
    };
    float2* sub = reinterpret_cast<float2*>(sh.L);
    if (b == 0) {
        if (tid == 0) sh.bad = 0;
        stage(sh.T, tile(0, 0));
        __syncthreads();
        for (int k = 0;; ++k) {
            ff_leaf(sh);
#pragma unroll
            for (int u = 0; u < 4 && on; ++u) tile(k, k)[hi * 32 + 4 * lo + u] = sh.T[hi][4 * lo + u];
            arrive(pivots);
            if (k == nt - 1) break;
            if (!wait_for(updates, (unsigned)(NW * k), updates, 0u, err)) return;
            stage(sh.A, tile(k + 1, k));
            float4 d[2] = {};
#pragma unroll
            for (int u = 0; u < 2 && on; ++u) d[u] = load4(tile(k + 1, k + 1), (2 * ty + u) * 16 + tx);
            arrive(panels);           // tile (k + 1, k) is read (the others' update overwrites it)
            if (on) {
                // L_k+1,k transposed: row hi, columns lo + 8 q; X_kk is lower triangular
                float s[4] = {}, e[4] = {};
#pragma unroll
                for (int m0 = 0; m0 < 32; m0 += 16) {
                    if (m0 <= hi)
#pragma unroll 4
                        for (int m = m0; m < m0 + 16; ++m)
#pragma unroll
                            for (int q = 0; q < 4; ++q) ff_fma_acc(s[q], e[q], sh.T[hi][m], sh.A[lo + 8 * q][m]);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 n = ff_norm(s[q], e[q]);
                        s[q] = n.x;
                        e[q] = n.y;
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) sub[hi * 32 + lo + 8 * q] = make_float2(s[q], e[q]);
            }
            __syncthreads();
            if (on) {
                update(sh.L, sh.L, d);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    sh.T[2 * ty + u][2 * tx] = make_float2(d[u].x, d[u].y);
                    sh.T[2 * ty + u][2 * tx + 1] = make_float2(d[u].z, d[u].w);
                }
            }
            __syncthreads();
        }
        if (tid == 0 && sh.bad) sync[0] = 1;
        return;
    }
    for (int k = 0; k < nt; ++k) {
        // the tiles of step k - 1 and this step's pivot
        if (!wait_for(updates, (unsigned)(NW * k), pivots, (unsigned)(k + 1), err)) return;
        // ---- panel
        if (b <= 4 * (nt - 1)) stage(sh.T, tile(k, k));
        for (int it = b - 1; it < 4 * (nt - 1); it += NW) {
            const int q = it & 3, below = nt - 1 - k, t = it >> 2;
            const bool is_l = t < below;
            // rows 8 q .. of A_ik, or columns 8 q .. of X_kj
            float2* src = is_l ? tile(k + 1 + t, k) : tile(k, t - below);
            if (!on) {
            } else if (is_l) sub[(tid >> 5) * 33 + (tid & 31)] = __ldcg(src + 256 * q + tid);
            else sub[tid] = __ldcg(src + hi * 32 + 8 * q + lo);
            __syncthreads();
            const float2* a = sub + (is_l ? 33 * lo : lo);
            const int step = is_l ? 1 : 8;
            if (on) {
                float s = 0.f, e = 0.f;
#pragma unroll
                for (int m0 = 0; m0 < 32; m0 += 16) {
#pragma unroll
                    for (int m = m0; m < m0 + 16; ++m) ff_fma_acc(s, e, sh.T[hi][m], a[m * step]);
                    const float2 n = ff_norm(s, e);
                    s = n.x;
                    e = n.y;
                }
                (is_l ? Lp + ((int64_t)(k + 1 + t) << 10) : src)[hi * 32 + 8 * q + lo] = make_float2(s, e);
            }
            __syncthreads();
        }
        if (k == nt - 1) return;
        arrive(panels);
        if (!wait_for(panels, (unsigned)(G * (k + 1)), updates, 0u, err)) return;
        // ---- update: row i = k + 1, .. has tiles j = i, .., 0; the first is block 0's
        const int tiles = nt * (nt + 1) / 2 - (k + 1) * (k + 2) / 2;
        int i = k + 1, j = i - b;
        float4 l[2], r[2], dn[2];     // operands, one tile ahead
        auto fetch = [&]() {
            while (j < 0) j += ++i + 1;
            const float2* Rg = j > k ? Lp + ((int64_t)j << 10) : tile(k, j);
            const float2* Lg = Lp + ((int64_t)i << 10);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                l[u] = load4(Lg, tid + 256 * u);
                r[u] = load4(Rg, tid + 256 * u);
                dn[u] = j == k ? make_float4(0.f, 0.f, 0.f, 0.f) : load4(tile(i, j), (2 * ty + u) * 16 + tx);
            }
        };
        if (on && b < tiles) fetch();
        for (int t = b; t < tiles; t += NW) {
            float2* D = tile(i, j);
            float4 d[2] = {dn[0], dn[1]};
            __syncthreads();          // the tile before is done with its operands
#pragma unroll
            for (int u = 0; u < 2 && on; ++u) {
                sh.L[tid + 256 * u] = l[u];
                sh.R[tid + 256 * u] = r[u];
            }
            __syncthreads();
            j -= NW;
            if (!on) continue;
            if (t + NW < tiles) fetch();
            update(sh.L, sh.R, d);
#pragma unroll
            for (int u = 0; u < 2; ++u) reinterpret_cast<float4*>(D)[(2 * ty + u) * 16 + tx] = d[u];
        }
        arrive(updates);
    }
}

__global__ void k_copy_add_diag(const double* __restrict__ src, double* __restrict__ dst,
                                int64_t s_pad, double nu) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= s_pad * s_pad) return;
    int64_t i = e / s_pad, j = e % s_pad;
    dst[e] = src[e] + ((i == j) ? nu : 0.0);
}

// What a float-float attempt takes from |M|_F, formed on the device so that the host
// need not wait for the norm: the shift nu = 2^-24 |M|_F (times 100 per retry),
// and 4^k and 2^k with |M|_F 4^k in [1, 4).
struct FFScale {
    double fro2, nu, up, out;
};

// The lower tiles of dst = (src + nu 100^attempt I) 4^k, row-major to 32 x 32 tiles
// (a block (32, 8) a tile); the pivots need both triangles of theirs. Over the whole
// square, each block forming the shift itself, 20 us at s_pad = 1024; now 12.
__global__ void k_copy_add_diag_ff(const double* __restrict__ src, float2* __restrict__ dst, int64_t s_pad,
                                   const FFScale* __restrict__ f, int attempt) {
    if (blockIdx.x > blockIdx.y) return;
    double nu = f->nu;
    for (int t = 0; t < attempt; ++t) nu *= 100.0;
    const double up = f->up;
    const int64_t j = (int64_t)blockIdx.x * 32 + threadIdx.x;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int64_t i = (int64_t)blockIdx.y * 32 + threadIdx.y + 8 * r;
        double v = src[i * s_pad + j];
        if (i == j) v += nu;
        dst[ff_tile_at(i, j, s_pad)] = ff_from_double(v * up);
    }
}

// L^{-1} = src 2^k from lower tiles: FP64 X, and FP32 B = X and Bt = X^T (null: not
// asked for), zeros above (below) the diagonal. A block (32, 8) per tile pair (i, j),
// (j, i): 11 us at s_pad = 1024, 22 as two kernels over rows.
__global__ void __launch_bounds__(256) k_ff_unpack(const float2* __restrict__ src, int64_t s_pad,
                                                   const FFScale* __restrict__ f, double* __restrict__ X,
                                                   float* __restrict__ B, float* __restrict__ Bt) {
    if (blockIdx.x > blockIdx.y) return;
    __shared__ float tile[32][33];
    const double out = f->out;
    const bool diag = blockIdx.x == blockIdx.y;
    const int64_t i0 = (int64_t)blockIdx.y * 32, j0 = (int64_t)blockIdx.x * 32;
    const int x = threadIdx.x;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int y = threadIdx.y + 8 * r;
        const int64_t at = (i0 + y) * s_pad + j0 + x, up = (j0 + y) * s_pad + i0 + x;
        const double v = diag && x > y ? 0.0 : ff_to_double(src[ff_tile_at(i0 + y, j0 + x, s_pad)]) * out;
        X[at] = v;
        if (!diag) X[up] = 0.0;
        if (B) {
            B[at] = (float)v;
            if (!diag) {
                B[up] = 0.f;
                Bt[at] = 0.f;
            }
            tile[y][x] = (float)v;
        }
    }
    if (!B) return;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int y = threadIdx.y + 8 * r;
        Bt[(j0 + y) * s_pad + i0 + x] = tile[x][y];
    }
}

// Frobenius norm^2 partials (single block, deterministic order).
// |M|_F^2 in two fixed-order stages: kFroBlocks block partials, then one
// block sums them.
constexpr int kFroBlocks = 128;

__global__ void __launch_bounds__(256) k_fro2_part(const double* __restrict__ M, int64_t m,
                                                  double* __restrict__ part) {
    __shared__ double red[8];
    double acc = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
        acc += M[e] * M[e];
    acc = msp::warp_sum(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += red[w];
        part[blockIdx.x] = v;
    }
}

__global__ void k_fro2_final(const double* __restrict__ part, FFScale* __restrict__ out) {
    double v = 0.0;
#pragma unroll
    for (int b = 0; b < kFroBlocks; b += 32) v += part[b + threadIdx.x];
    v = msp::warp_sum(v);
    if (threadIdx.x == 0) {
        const double fn = sqrt(v);
        const int k = fn > 0.0 && isfinite(fn) ? -(ilogb(fn) / 2) : 0;
        *out = FFScale{v, ldexp(1.0, -24) * fn, ldexp(1.0, 2 * k), ldexp(1.0, k)};
    }
}

template <typename T>
__global__ void k_cast_tri(const double* __restrict__ X, T* __restrict__ B, T* __restrict__ Bt,
                           int64_t s_pad) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= s_pad * s_pad) return;
    int64_t i = e / s_pad, j = e % s_pad;
    double v = (j <= i) ? X[e] : 0.0;
    B[e] = (T)v;
    Bt[j * s_pad + i] = (T)v;
}

template <int TS>
void launch_dgemm_ts(msp_ctx* ctx, bool ta, bool tb, int64_t m, int64_t n, int64_t k, double alpha,
                     const double* A, int64_t lda, const double* B, int64_t ldb, double beta,
                     double* Cm, int64_t ldc, int tri_a, int tri_b, int lower_out) {
    dim3 grid((unsigned)((n + TS - 1) / TS), (unsigned)((m + TS - 1) / TS));
    if (!ta && !tb) k_dgemm<false, false, TS><<<grid, 256, 0, ctx->stream>>>(m, n, k, alpha, A, lda, B, ldb, beta, Cm, ldc, tri_a, tri_b, lower_out);
    else if (!ta && tb) k_dgemm<false, true, TS><<<grid, 256, 0, ctx->stream>>>(m, n, k, alpha, A, lda, B, ldb, beta, Cm, ldc, tri_a, tri_b, lower_out);
    else if (ta && !tb) k_dgemm<true, false, TS><<<grid, 256, 0, ctx->stream>>>(m, n, k, alpha, A, lda, B, ldb, beta, Cm, ldc, tri_a, tri_b, lower_out);
    else k_dgemm<true, true, TS><<<grid, 256, 0, ctx->stream>>>(m, n, k, alpha, A, lda, B, ldb, beta, Cm, ldc, tri_a, tri_b, lower_out);
}

msp_status dgemm(msp_ctx* ctx, bool ta, bool tb, int64_t m, int64_t n, int64_t k, double alpha,
                 const double* A, int64_t lda, const double* B, int64_t ldb, double beta,
                 double* Cm, int64_t ldc, int tri_a = 0, int tri_b = 0, int lower_out = 0) {
    // FP64 work is pipe-bound on this part: prefer the larger tile only when it
    // still yields two blocks per SM
    const int64_t tiles32 = ((m + 31) / 32) * ((n + 31) / 32);
    if (tiles32 >= 2 * ctx->num_sms)
        launch_dgemm_ts<32>(ctx, ta, tb, m, n, k, alpha, A, lda, B, ldb, beta, Cm, ldc, tri_a, tri_b, lower_out);
    else
        launch_dgemm_ts<16>(ctx, ta, tb, m, n, k, alpha, A, lda, B, ldb, beta, Cm, ldc, tri_a, tri_b, lower_out);
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

msp_status leaf(msp_ctx* ctx, double* M, double* X, int64_t ld, int64_t n, int* fail) {
    // set once per device; batch set-up calls this from several threads
    static std::atomic<bool> attr_set[64];
    const int d = ctx->device;
    if (d < 0 || d >= 64 || !attr_set[d].load()) {
        MSP_CUDA_TRY(ctx, cudaFuncSetAttribute(k_chol_leaf, cudaFuncAttributeMaxDynamicSharedMemorySize, kLeafSmem));
        if (d >= 0 && d < 64) attr_set[d] = true;
    }
    k_chol_leaf<<<1, kLeafThreads, kLeafSmem, ctx->stream>>>(M, X, ld, (int)n, fail);
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

// Recursive Cholesky + inverse of the n x n block at offset `off` of M (ld),
// inverse into X (same offsets); T1/T2 are n x n temporaries (ld). Only X =
// L^{-1} is kept: M is scratch (the Schur complements overwrite its lower
// triangle, the leaves leave their L blocks there, L21 is not stored). Leaves
// of at most 32: a leaf runs on one SM, whose FP64 pipe bounds it (its work
// grows as nb^3), while the products of the recursion spread over all SMs.
msp_status chol_inv(msp_ctx* ctx, double* M, double* X, double* T1, double* T2, int64_t ld, int64_t off,
                    int64_t n, int* fail, int depth) {
    if (n <= 32) return leaf(ctx, M + off * ld + off, X + off * ld + off, ld, n, fail);
    int64_t n1 = std::max<int64_t>(32, (n / 2) / 32 * 32);
    int64_t n2 = n - n1;
    double* A21 = M + (off + n1) * ld + off;
    double* A22 = M + (off + n1) * ld + off + n1;
    double* X11 = X + off * ld + off;
    double* X21 = X + (off + n1) * ld + off;
    double* X22 = X + (off + n1) * ld + off + n1;
    MSP_TRY(chol_inv(ctx, M, X, T1, T2, ld, off, n1, fail, depth + 1));
    // T1 = L21 = A21 X11^T   (n2 x n1; X11^T is upper triangular)
    MSP_TRY(dgemm(ctx, false, true, n2, n1, n1, 1.0, A21, ld, X11, ld, 0.0, T1, ld, 0, 1, 0));
    // T2 = L21 X11 (X11 lower) needs only T1 and X11, so it runs on the side
    // stream of this depth while A22 is updated and factored on the main
    // stream. Disjoint memory: T1 and T2 hold columns [0, n1) of the
    // temporaries, the second half works in columns [n1, n) of them.
    // The stream and both events of this depth are the context's (created
    // once): recursion at one depth is sequential, and every wait on an
    // event is enqueued before the event is recorded again.
    cudaStream_t side = nullptr;
    cudaEvent_t ev_t1 = nullptr, ev_t2 = nullptr;
    if (ctx->fac_overlap && depth < 8) {
        cudaEvent_t* ev = ctx->fac_ev[depth];
        if ((ctx->fac_side[depth] ||
             cudaStreamCreateWithFlags(&ctx->fac_side[depth], cudaStreamNonBlocking) == cudaSuccess) &&
            (ev[0] || cudaEventCreateWithFlags(&ev[0], cudaEventDisableTiming) == cudaSuccess) &&
            (ev[1] || cudaEventCreateWithFlags(&ev[1], cudaEventDisableTiming) == cudaSuccess)) {
            side = ctx->fac_side[depth];
            ev_t1 = ev[0];
            ev_t2 = ev[1];
        }
    }
    if (side && (cudaEventRecord(ev_t1, ctx->stream) != cudaSuccess ||
                 cudaStreamWaitEvent(side, ev_t1, 0) != cudaSuccess)) {
        cudaGetLastError();
        side = nullptr;     // fall back to the main stream
    }
    if (!side) cudaGetLastError();
    msp_status st = MSP_OK;
    if (side) {
        cudaStream_t main_stream = ctx->stream;
        ctx->stream = side;
        st = dgemm(ctx, false, false, n2, n1, n1, 1.0, T1, ld, X11, ld, 0.0, T2, ld, 0, 2, 0);
        ctx->stream = main_stream;
        if (st == MSP_OK && cudaEventRecord(ev_t2, side) != cudaSuccess)
            st = msp_set_error(ctx, MSP_ECUDA, "factor: side stream record failed");
    }
    // A22 -= L21 L21^T (lower triangle is all the recursion reads)
    if (st == MSP_OK)
        st = dgemm(ctx, false, true, n2, n2, n1, -1.0, T1, ld, T1, ld, 1.0, A22, ld, 0, 0, 1);
    if (st == MSP_OK) st = chol_inv(ctx, M, X, T1 + n1, T2 + n1, ld, off + n1, n2, fail, depth + 1);
    if (st == MSP_OK) {
        if (side) {
            if (cudaStreamWaitEvent(ctx->stream, ev_t2, 0) != cudaSuccess)
                st = msp_set_error(ctx, MSP_ECUDA, "factor: side stream join failed");
        } else {
            st = dgemm(ctx, false, false, n2, n1, n1, 1.0, T1, ld, X11, ld, 0.0, T2, ld, 0, 2, 0);
        }
    }
    if (side && st != MSP_OK) cudaStreamSynchronize(side);
    MSP_TRY(st);
    // X21 = -X22 T2 (X22 lower)
    MSP_TRY(dgemm(ctx, false, false, n2, n1, n2, -1.0, X22, ld, T2, ld, 0.0, X21, ld, 1, 0, 0));
    return MSP_OK;
}

// One float-float attempt: k_chol_inv_ff on as many blocks as its widest step has
// work for and one more, one an SM at most. sync: six words, see there.
msp_status chol_inv_ff(msp_ctx* ctx, float2* S, float2* Lp, int64_t sp, int* sync) {
    int nt = (int)(sp / 32), per_sm = 0;
    MSP_CUDA_TRY(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_chol_inv_ff, kFFThreads, 0));
    if (per_sm < 1) return msp_set_error(ctx, MSP_ECUDA, "factor: kernel does not fit on an SM");
    const int work = std::max(nt * (nt + 1) / 2 - 1, 4 * (nt - 1));
    const int grid = std::max(2, std::min(work + 1, ctx->num_sms));
    void* args[] = {&S, &Lp, &nt, &sync};
    ++ctx->launches;
    MSP_CUDA_TRY(ctx, cudaLaunchCooperativeKernel((const void*)k_chol_inv_ff, dim3(grid), dim3(kFFThreads), args, 0,
                                                  ctx->stream));
    return MSP_OK;
}

// Cholesky inverse of M + nu I (lower L^{-1} into Linv64), s_pad x s_pad
// FP64 M with identity padding. FP32 data: M carries rounding errors of
// about 2^-24 |M|_F (its operands are FP32), which leave it indefinite by
// that much where it has tiny eigenvalues; nu starts there, which saves a
// second factorisation. FP64 data: unshifted first, then s 2^-52 |M|_F.
// Then nu x 100 per retry, at most 4 retries, else MSP_ENOTPD.
msp_status factor_shifted(msp_ctx* ctx, const double* M, int64_t s, int64_t sp, bool fp32_data,
                          double* Linv64, double* shift_out, int* retries_out, float* B = nullptr,
                          float* Bt = nullptr) {
    // FP32 data: the factorisation in float-float (its backward error, a
    // small multiple of s 2^-46 |M|, stays far below the shift 2^-24 |M|_F
    // the data needs), on M scaled by a power of four to |M|_F in [1, 4) so
    // that no float range limit is near
    const bool ff = fp32_data && ctx->factor_ff;
    void* scr = nullptr;
    size_t mat = (size_t)sp * sp * 8;
    MSP_TRY(msp_scratch(ctx, (ff ? mat + (size_t)sp * 32 * 8 : 3 * mat) + 2048, &scr));
    double* Mw = (double*)scr;
    double* T1 = Mw + sp * sp;                       // ff: 32 columns, the panel
    double* T2 = T1 + sp * sp;
    int* fail = (int*)(ff ? T1 + 32 * sp : T2 + sp * sp);        // and, ff, the words of k_chol_inv_ff
    FFScale* fro = (FFScale*)(fail + 16);
    double* fro_part = (double*)(fro + 1);
    int* hflag = (int*)ctx->host_flags;
    double* hfro = (double*)((char*)ctx->host_flags + 128);
    auto fro_launch = [&]() -> msp_status {
        k_fro2_part<<<kFroBlocks, 256, 0, ctx->stream>>>(M, sp * sp, fro_part);
        MSP_CHECK_LAUNCH(ctx);
        k_fro2_final<<<1, 32, 0, ctx->stream>>>(fro_part, fro);
        MSP_CHECK_LAUNCH(ctx);
        MSP_CUDA_TRY(ctx, cudaMemcpyAsync(hfro, &fro->fro2, 8, cudaMemcpyDeviceToHost, ctx->stream));
        return MSP_OK;
    };
    auto fro_norm = [&](double* out) -> msp_status {
        MSP_TRY(fro_launch());
        MSP_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
        *out = std::sqrt(*hfro);
        return MSP_OK;
    };
    double nu = 0.0;
    if (ff) {
        // nu and the scaling are formed on the device (FFScale); the host reads the
        // norm with the outcome
        MSP_TRY(fro_launch());
    } else if (fp32_data) {
        double fn = 0.0;
        MSP_TRY(fro_norm(&fn));
        nu = std::ldexp(1.0, -24) * fn;
    }
    for (int attempt = 0; attempt <= 4; ++attempt) {
        unsigned blocks = (unsigned)((sp * sp + 255) / 256);
        MSP_CUDA_TRY(ctx, cudaMemsetAsync(fail, 0, 6 * sizeof(int), ctx->stream));
        if (ff) {
            const dim3 tiles((unsigned)(sp / 32), (unsigned)(sp / 32)), thr(32, 8);
            k_copy_add_diag_ff<<<tiles, thr, 0, ctx->stream>>>(M, reinterpret_cast<float2*>(Mw), sp, fro, attempt);
            MSP_CHECK_LAUNCH(ctx);
            MSP_TRY(chol_inv_ff(ctx, reinterpret_cast<float2*>(Mw), reinterpret_cast<float2*>(T1), sp, fail));
            k_ff_unpack<<<tiles, thr, 0, ctx->stream>>>(reinterpret_cast<float2*>(Mw), sp, fro, Linv64, B, Bt);
            MSP_CHECK_LAUNCH(ctx);
        } else {
            k_copy_add_diag<<<blocks, 256, 0, ctx->stream>>>(M, Mw, sp, nu);
            MSP_CHECK_LAUNCH(ctx);
            MSP_CUDA_TRY(ctx, cudaMemsetAsync(Linv64, 0, mat, ctx->stream));
            MSP_TRY(chol_inv(ctx, Mw, Linv64, T1, T2, sp, 0, sp, fail, 0));
        }
        MSP_CUDA_TRY(ctx, cudaMemcpyAsync(hflag, fail, 3 * sizeof(int), cudaMemcpyDeviceToHost,
                                          ctx->stream));
        MSP_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
        if (hflag[2]) return msp_set_error(ctx, (msp_status)hflag[2], "factor: grid barrier timed out");
        if (ff && attempt == 0) nu = std::ldexp(1.0, -24) * std::sqrt(*hfro);
        if (hflag[0] == 0) {
            *shift_out = nu;
            *retries_out = attempt;
            return MSP_OK;
        }
        if (nu == 0.0) {
            double fn = 0.0;
            MSP_TRY(fro_norm(&fn));
            nu = (fp32_data ? std::ldexp(1.0, -24) : (double)s * std::ldexp(1.0, -52)) * fn;
            if (nu == 0.0) break;
        } else {
            nu *= 100.0;
        }
    }
    return msp_set_error(ctx, MSP_ENOTPD,
                         "matrix + shift is not positive definite after 4 retries (last shift %g)",
                         nu / 100.0);
}

}  // namespace

// W symmetrised, and its FP64 copy.
msp_status msp_symmetrize_w(msp_ctx* ctx, msp_factor_s* f) {
    const int64_t sp = f->s_pad;
    const dim3 blk(32, 32), grid((unsigned)((sp + 31) / 32), (unsigned)((sp + 31) / 32));
    if (f->dtype == MSP_F32)
        k_symmetrize<float><<<grid, blk, 0, ctx->stream>>>((float*)f->W, f->W64, sp);
    else
        k_symmetrize<double><<<grid, blk, 0, ctx->stream>>>((double*)f->W, f->W64, sp);
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

// Build M2, its shifted Cholesky inverse, and the working copies B, Bt. `Ct` is C~
// (phi_rows x s_pad, dtype of the sketch); W symmetrised, by w_ready.
msp_status msp_build_factor(msp_ctx* ctx, msp_factor_s* f, const void* Ct, int64_t phi_rows, cudaEvent_t w_ready) {
    const int64_t sp = f->s_pad;
    // M2 = Ct^T Ct + lam_t W: on the tensor cores (FP32 data), else split-K
    // partial Grams (upper tiles, mirrored) then the fixed-order FP64
    // combination
    if (f->dtype == MSP_F32 && ctx->gram_tc && msp_gram_tc_ok(sp)) {
        MSP_TRY(msp_gram_tc(ctx, (const float*)Ct, phi_rows, sp, f->s, sp, (const float*)f->W, f->lam_tilde, f->M2,
                            w_ready));
    } else {
        if (w_ready) MSP_CUDA_TRY(ctx, cudaStreamWaitEvent(ctx->stream, w_ready, 0));
        double* P = nullptr;
        int slices = 0;
        const unsigned fb = (unsigned)((sp * sp + 255) / 256);
        if (f->dtype == MSP_F32) {
            MSP_TRY(launch_gram(ctx, (const float*)Ct, phi_rows, sp, f->s, sp, 0, &P, &slices));
            k_gram_finish<float><<<fb, 256, 0, ctx->stream>>>(P, slices, (const float*)f->W, f->lam_tilde,
                                                               f->s, sp, f->M2);
        } else {
            MSP_TRY(launch_gram(ctx, (const double*)Ct, phi_rows, sp, f->s, sp, 0, &P, &slices));
            k_gram_finish<double><<<fb, 256, 0, ctx->stream>>>(P, slices, (const double*)f->W, f->lam_tilde,
                                                                f->s, sp, f->M2);
        }
        MSP_CHECK_LAUNCH(ctx);
    }
    const bool f32 = f->dtype == MSP_F32;
    MSP_TRY(factor_shifted(ctx, f->M2, f->s, sp, f32, f->Linv64, &f->shift, &f->retries,
                           f32 ? (float*)f->B : nullptr, f32 ? (float*)f->Bt : nullptr));
    if (f32 && ctx->factor_ff) return MSP_OK;       // B and Bt are there
    unsigned b2 = (unsigned)((sp * sp + 255) / 256);
    if (f32)
        k_cast_tri<float><<<b2, 256, 0, ctx->stream>>>(f->Linv64, (float*)f->B, (float*)f->Bt, sp);
    else
        k_cast_tri<double><<<b2, 256, 0, ctx->stream>>>(f->Linv64, (double*)f->B, (double*)f->Bt, sp);
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

namespace {

// hi = fl32(src), lo = fl32(src - hi)
__global__ void k_split_pair(const double* __restrict__ src, float* __restrict__ hi, float* __restrict__ lo,
                             int64_t count) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= count) return;
    const float h = (float)src[e];
    hi[e] = h;
    lo[e] = (float)(src[e] - (double)h);
}

}  // namespace

// The level-2 operator H = C^T C + lam~ W of a sketched level 2, its Gram
// accumulated as M2's on the FP32 pipe (compensated; FP64 for FP64 data), so that
// products with it are no further from C^T (C d) + lam~ W d, relative to |C|^2 |d|, than
// the passes over C in the working precision are. (Along directions that C nearly
// annihilates the passes are closer. It shows in the level-1 iterations: 52.0 with them and
// 53.9 with H on FP64 systems of n 500 to 700 with outliers of 1e4; 346 and 347 on FP32
// kernel systems of n 1000 to 5900.) One Gram of n rows (0.1 ms at n = 5000, s = 312)
// against a pass over C and two grid barriers saved in every level-2 iteration.
msp_status msp_form_level2(msp_ctx* ctx, msp_factor_s* f, const void* C, int64_t n) {
    const int64_t sp = f->s_pad, mat = sp * sp;
    const unsigned fb = (unsigned)((mat + 255) / 256);
    MSP_TRY(msp_alloc(ctx, &f->H, (size_t)mat * 8));
    double* P = nullptr;
    int slices = 0;
    if (f->dtype == MSP_F32) {
        MSP_TRY(launch_gram(ctx, (const float*)C, n, sp, f->s, sp, mat, &P, &slices));
        double* H64 = P + slices * mat;
        k_gram_finish<float><<<fb, 256, 0, ctx->stream>>>(P, slices, (const float*)f->W, f->lam_tilde, f->s, sp, H64);
        MSP_CHECK_LAUNCH(ctx);
        k_split_pair<<<fb, 256, 0, ctx->stream>>>(H64, (float*)f->H, (float*)f->H + mat, mat);
    } else {
        MSP_TRY(launch_gram(ctx, (const double*)C, n, sp, f->s, sp, 0, &P, &slices));
        k_gram_finish<double><<<fb, 256, 0, ctx->stream>>>(P, slices, (const double*)f->W, f->lam_tilde, f->s, sp,
                                                            (double*)f->H);
    }
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

// G64 = X^T X + diag I over the leading s columns of X (rows x ld FP32
// row-major, columns s..s_pad-1 zero): split-K partial Grams with compensated
// FP32 sums, combined in FP64 in a fixed order; pad block identity.
msp_status msp_gram64(msp_ctx* ctx, const float* X, int64_t rows, int64_t ld, int64_t s, int64_t sp,
                      double diag, double* G64) {
    double* P = nullptr;
    int slices = 0;
    MSP_TRY(launch_gram(ctx, X, rows, ld, s, sp, 0, &P, &slices));
    k_gram_finish<float><<<(unsigned)((sp * sp + 255) / 256), 256, 0, ctx->stream>>>(
        P, slices, (const float*)nullptr, diag, s, sp, G64);
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

// Minv = M^{-1} (dense FP64) for an SPD s_pad x s_pad M64: FP64 Cholesky,
// shifted only on failure (the FP64-data rule), then L^{-T} L^{-1}.
msp_status msp_spd_inverse(msp_ctx* ctx, const double* M64, int64_t s, int64_t sp, double* Linv64,
                           double* Minv, double* shift, int* retries) {
    MSP_TRY(factor_shifted(ctx, M64, s, sp, false, Linv64, shift, retries));
    return dgemm(ctx, true, false, sp, sp, sp, 1.0, Linv64, sp, Linv64, sp, 0.0, Minv, sp);
}

// Dense inverse of G + diag I with G = X^T X. G is the Gram of the stored
// FP32 X itself, accumulated with compensated FP32 partial sums combined in
// FP64: PSD to about 2^-48 relative, so the FP64-data shift rule (unshifted
// first) applies. An FP32 copy of the inverse would perturb its products by
// about 2^-24 kappa(G), so the inverse stays FP64. G64 receives G + diag I.
msp_status msp_gram_inverse(msp_ctx* ctx, const float* X, int64_t rows, int64_t s, int64_t sp,
                            double diag, double* G64, double* Linv64, double* Minv,
                            double* shift, int* retries) {
    MSP_TRY(msp_gram64(ctx, X, rows, sp, s, sp, diag, G64));
    return msp_spd_inverse(ctx, G64, s, sp, Linv64, Minv, shift, retries);
}

namespace {

// Partial products P[slice][a][b] = sum_{k in slice} X[k][a] Y[k][b] for one
// 64 x 64 output tile (blockIdx.x over tile pairs, blockIdx.y the K slice),
// FP32 chunks of 16 accumulated with TwoSum into FP64 outputs. Columns of X
// at or beyond ncx (of Y: ncy) read as zero.
__global__ void __launch_bounds__(256, 4) k_gemm_tn(const float* __restrict__ X, int64_t ldx, int64_t ncx,
                                                   const float* __restrict__ Y, int64_t ldy, int64_t ncy,
                                                   int64_t K, int64_t ny_pad, int64_t nx_pad,
                                                   double* __restrict__ P) {
    __shared__ __align__(16) float As[16][64];
    __shared__ __align__(16) float Bs[16][64];
    const int nty = (int)(ny_pad / 64);
    const int ta = blockIdx.x / nty, tb = blockIdx.x % nty;
    const int64_t a0 = (int64_t)ta * 64, b0 = (int64_t)tb * 64;
    const int64_t kper = ((K + gridDim.y - 1) / gridDim.y + 15) / 16 * 16;
    const int64_t kbeg = (int64_t)blockIdx.y * kper;
    const int64_t kend = min(K, kbeg + kper);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float hi[4][4], lo[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { hi[i][j] = 0.f; lo[i][j] = 0.f; }
    for (int64_t k0 = kbeg; k0 < kend; k0 += 16) {
        for (int e = threadIdx.x; e < 16 * 64; e += 256) {
            const int kk = e >> 6, cc = e & 63;
            const bool in = (k0 + kk) < kend;
            As[kk][cc] = (in && a0 + cc < ncx) ? X[(k0 + kk) * ldx + a0 + cc] : 0.f;
            Bs[kk][cc] = (in && b0 + cc < ncy) ? Y[(k0 + kk) * ldy + b0 + cc] : 0.f;
        }
        __syncthreads();
        float acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            const float4 va = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
            const float4 vb = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
            const float av[4] = {va.x, va.y, va.z, va.w}, bv[4] = {vb.x, vb.y, vb.z, vb.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) two_sum_add(hi[i][j], lo[i][j], acc[i][j]);
        __syncthreads();
    }
    double* Ps = P + (int64_t)blockIdx.y * nx_pad * ny_pad;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            Ps[(a0 + ty * 4 + i) * ny_pad + b0 + tx * 4 + j] = (double)hi[i][j] + (double)lo[i][j];
}

__global__ void k_sum_slices_f32(const double* __restrict__ P, int64_t len, float* __restrict__ out) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= len) return;
    double v = 0.0;
#pragma unroll
    for (int sl = 0; sl < kGemmSlices; ++sl) v += P[(int64_t)sl * len + e];
    out[e] = (float)v;
}

}  // namespace

// C = X^T Y (FP32 nx_pad x ny_pad row-major, nx_pad and ny_pad multiples of
// 64) for X: K x ncx (ldx) and Y: K x ncy (ldy), FP32 row-major; entries past
// ncx / ncy are zero. Compensated FP32 chunk sums combined in FP64, rounded
// once to FP32.
msp_status msp_gemm_tn(msp_ctx* ctx, const float* X, int64_t ldx, int64_t ncx, const float* Y, int64_t ldy,
                       int64_t ncy, int64_t K, int64_t nx_pad, int64_t ny_pad, float* C) {
    void* scr = nullptr;
    MSP_TRY(msp_scratch(ctx, (size_t)kGemmSlices * nx_pad * ny_pad * 8, &scr));
    double* P = (double*)scr;
    dim3 grid((unsigned)((nx_pad / 64) * (ny_pad / 64)), kGemmSlices);
    k_gemm_tn<<<grid, 256, 0, ctx->stream>>>(X, ldx, ncx, Y, ldy, ncy, K, ny_pad, nx_pad, P);
    MSP_CHECK_LAUNCH(ctx);
    const int64_t len = nx_pad * ny_pad;
    k_sum_slices_f32<<<(unsigned)((len + 255) / 256), 256, 0, ctx->stream>>>(P, len, C);
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

// The wait limit of this unit's kernel (k_chol_inv_ff) on the current device; 0 restores
// the default.
msp_status msp_grid_wait_limit_factor(msp_ctx* ctx, unsigned long long ns) {
    const unsigned long long v = ns ? ns : msp::kWaitLimitNs;
    MSP_CUDA_TRY(ctx, cudaMemcpyToSymbol(msp::g_grid_wait_limit_ns, &v, sizeof v));
    return MSP_OK;
}

extern "C" msp_status msp_set_factor_float_float(msp_ctx* ctx, int on) {
    if (!ctx) return msp_set_error(nullptr, MSP_EINVAL, "ctx is NULL");
    ctx->factor_ff = on != 0;
    return MSP_OK;
}
