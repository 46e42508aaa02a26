// Level-1 and level-2 iterations of MSP on sm_103a (Algorithm 1 step 5 and
// Algorithm 2).
//
// One level-1 (outer) iteration is two launches:
//   k_gemv      q = (A + lam I) p, one pass over A, with the dot p^T q fused;
//               the last block to finish forms alpha = (r^T z) / (p^T q).
//               (With packed tiles k_symv_packed of symv.cu: it also forms the
//               direction p = w + beta p, and leaves p^T q in block partials.)
//   k_level2    persistent cooperative kernel: x += alpha p, r -= alpha q,
//               convergence test on |r|, then SolveM1(r) (Algorithm 2):
//               g = C^T r; level-2 PCG on (C^T C + lam~ W) y = g
//               preconditioned by M2^{-1} v = B^T (B v); w = (r - C y)/lam~;
//               finally the flexible (Polak-Ribiere) beta and p = w + beta p.
// Level-2 vectors (length s) are held redundantly in every block's shared
// memory; every block computes the same scalars from the same partial sums
// in the same order, so all blocks take identical branches and the number of
// grid barriers always matches. Reductions use fixed orders (deterministic).
#include "bulk.cuh"
#include "l2_columns.cuh"
#include "msp_internal.cuh"

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>

namespace {

constexpr int kNW = 16;            // warps per block in k_level2
constexpr int kThreads = kNW * 32;
constexpr int kRowChunk = kThreads;          // rows of C whose r, w are staged at a time
constexpr int kQScratch = 4 * kNW * 32;      // slot sums of the level-1 update

enum { MODE_INIT = 0, MODE_ITER = 1, MODE_APPLY = 2 };
enum { PHASE_ALL = 0, PHASE_FRONT = 1, PHASE_BACK = 2 };

template <typename T> struct Vec16;
template <> struct Vec16<float> { using type = float4; static constexpr int W = 4; };
template <> struct Vec16<double> { using type = double2; static constexpr int W = 2; };

template <typename T>
__device__ inline void load16(const T* p, T* out) {
    typename Vec16<T>::type v = *reinterpret_cast<const typename Vec16<T>::type*>(p);
    if constexpr (Vec16<T>::W == 4) { out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w; }
    else { out[0] = v.x; out[1] = v.y; }
}

// One vector load of a row slice: 16 bytes of FP32 / FP64, or 8 bytes of
// BF16 (4 values, widened to FP32 exactly), so that every storage type puts
// the same 4 (FP64: 2) consecutive values in each lane step.
template <typename T>
__device__ inline void load_vec(const T* p, T* out) { load16(p, out); }
__device__ inline void load_vec(const __nv_bfloat16* p, float* out) {
    const uint2 v = *reinterpret_cast<const uint2*>(p);
    out[0] = __uint_as_float(v.x << 16);
    out[1] = __uint_as_float(v.x & 0xFFFF0000u);
    out[2] = __uint_as_float(v.y << 16);
    out[3] = __uint_as_float(v.y & 0xFFFF0000u);
}

// Values per vector load of a storage type.
template <typename TS> struct StoreW { static constexpr int W = 16 / (int)sizeof(TS); };
template <> struct StoreW<__nv_bfloat16> { static constexpr int W = 4; };

// Streaming (evict-first) 16-byte load: A is read once per pass, so it should
// not displace the sketch C, which the level-2 iteration re-reads from L2.
template <typename T>
__device__ inline void load16_stream(const T* p, T* out) {
    typename Vec16<T>::type v = __ldcs(reinterpret_cast<const typename Vec16<T>::type*>(p));
    if constexpr (Vec16<T>::W == 4) { out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w; }
    else { out[0] = v.x; out[1] = v.y; }
}

// Deterministic block-wide sum of one double per thread (all threads get it).
__device__ inline double block_sum(double v, double* red) {
    v = msp::warp_sum(v);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    double t = 0.0;
    const int nw = blockDim.x >> 5;
    for (int k = 0; k < nw; ++k) t += red[k];
    return t;
}

// Sum of a per-block partial array in fixed order (all threads get it).
__device__ inline double sum_parts(const double* parts, int stride, int G, double* red) {
    double v = 0.0;
    for (int k = threadIdx.x; k < G; k += blockDim.x) v += __ldcg(&parts[(int64_t)k * stride]);
    return block_sum(v, red);
}

// Two block sums at once (red holds 64 doubles): per value the order of
// block_sum, with one pair of barriers.
__device__ inline void block_sum2(double& v0, double& v1, double* red) {
    v0 = msp::warp_sum(v0);
    v1 = msp::warp_sum(v1);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) {
        red[w] = v0;
        red[32 + w] = v1;
    }
    __syncthreads();
    double t0 = 0.0, t1 = 0.0;
    const int nw = blockDim.x >> 5;
    for (int k = 0; k < nw; ++k) {
        t0 += red[k];
        t1 += red[32 + k];
    }
    v0 = t0;
    v1 = t1;
}

// sum_parts of the entries at offsets o0 and o1 of every block's record.
__device__ inline void sum_parts2(const double* parts, int stride, int G, double* red, double& s0, double& s1) {
    double v0 = 0.0, v1 = 0.0;
    for (int k = threadIdx.x; k < G; k += blockDim.x) {
        v0 += __ldcg(&parts[(int64_t)k * stride]);
        v1 += __ldcg(&parts[(int64_t)k * stride + 1]);
    }
    block_sum2(v0, v1, red);
    s0 = v0;
    s1 = v1;
}

// ------------------------------------------------------------------ GEMV

// q = (A + lam I) p; warp per row (grid-stride); lane reads 16 B vectors.
// The block partials of p^T q are combined by the last block, which writes
// ctl->pq and ctl->alpha = ctl->rz / pq (or flags an error).
template <typename TA, typename T, bool VEC>
__global__ void __launch_bounds__(256) k_gemv(const TA* __restrict__ A, int64_t lda, int64_t n,
                                             double lam, const T* __restrict__ p,
                                             T* __restrict__ q, double* __restrict__ part,
                                             CtlBlock* ctl) {
    if (ctl->done | ctl->error) return;
    __shared__ double red[32];
    __shared__ bool am_last;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    double pq = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n;
         i += warps) {
        const TA* row = A + i * lda;
        T acc = T(0);
        if constexpr (VEC) {
            constexpr int W = Vec16<TA>::W;
            int64_t j = (int64_t)lane * W;
            // 4 independent 16 B loads in flight per lane
            for (; j + 3 * 32 * W < n; j += 4 * 32 * W) {
                TA a[4][W];
                T pv[4][W];
#pragma unroll
                for (int u = 0; u < 4; ++u) load16_stream(row + j + u * 32 * W, a[u]);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
#pragma unroll
                    for (int e = 0; e < W; ++e) pv[u][e] = p[j + u * 32 * W + e];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int e = 0; e < W; ++e) acc += (T)a[u][e] * pv[u][e];
            }
            for (; j < n; j += 32 * W) {
                TA a[W];
                load16_stream(row + j, a);
#pragma unroll
                for (int e = 0; e < W; ++e) acc += (T)a[e] * p[j + e];
            }
        } else {
            for (int64_t j = lane; j < n; j += 32) acc += (T)__ldcs(&row[j]) * p[j];
        }
        acc = msp::warp_sum(acc);
        if (lane == 0) {
            T qi = acc + (T)lam * p[i];
            q[i] = qi;
            pq += (double)p[i] * (double)qi;
        }
    }
    double tot = block_sum(pq, red);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = tot;
        __threadfence();
        unsigned int t = atomicAdd(&ctl->last_block_counter, 1u);
        am_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    double all = sum_parts(part, 1, gridDim.x, red);
    if (threadIdx.x == 0) {
        ctl->last_block_counter = 0;
        ctl->pq = all;
        if (!isfinite(all)) { ctl->error = MSP_ENONFINITE; }
        else if (!(all > 0.0)) { ctl->error = MSP_ENOTPD; }
        else ctl->alpha = ctl->rz / all;
    }
}

// Exact binary32 -> binary64 widening with integer instructions (the FP64
// pipe, which bounds the residual, then only executes the FMAs). Subnormal
// inputs are flushed to zero (their products are below 1e-37 |x|); infinities
// and NaNs keep their class.
__device__ inline double widen_f32(float f) {
    const uint32_t u = __float_as_uint(f);
    const uint32_t ex = u & 0x7f800000u;
    const uint64_t sign = (uint64_t)(u & 0x80000000u) << 32;
    uint64_t bits;
    if (ex == 0u) bits = sign;                                               // zero / subnormal
    else if (ex == 0x7f800000u) bits = sign | 0x7ff0000000000000ull | ((uint64_t)(u & 0x007fffffu) << 29);
    else bits = sign | (((uint64_t)(u & 0x7fffffffu) << 29) + ((uint64_t)(1023 - 127) << 52));
    return __longlong_as_double((long long)bits);
}

// A entry widened to FP64 (exact for every storage type).
__device__ inline double wide64(double v) { return v; }
__device__ inline double wide64(float v) { return (double)v; }
__device__ inline double wide64(__nv_bfloat16 v) { return (double)__bfloat162float(v); }

// out = b - (A + lam I) x  (or (A + lam I) x if b == nullptr), FP64
// accumulation; |out|^2 into *norm2 (last block, fixed order). The FP64 FMA
// rate bounds this kernel on this part (two FMAs per clock per SM): loads are
// vectorised (16 B of A, 32 B of x per lane step) and A is widened with
// integer instructions so that the FP64 pipe issues only the FMAs.
template <typename TA, bool VEC>
__global__ void __launch_bounds__(256) k_matvec64(const TA* __restrict__ A, int64_t lda, int64_t n,
                                                 double lam, const double* __restrict__ x,
                                                 const double* __restrict__ b,
                                                 double* __restrict__ out, double* __restrict__ part,
                                                 unsigned int* counter, double* norm2) {
    __shared__ double red[32];
    __shared__ bool am_last;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    double nn = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n;
         i += warps) {
        const TA* row = A + i * lda;
        double acc0 = 0.0, acc1 = 0.0;
        if constexpr (VEC && sizeof(TA) == 4) {
            int64_t j = (int64_t)lane * 4;
            for (; j + 32 * 4 < n; j += 2 * 32 * 4) {
                const float4 a0 = __ldcs(reinterpret_cast<const float4*>(row + j));
                const float4 a1 = __ldcs(reinterpret_cast<const float4*>(row + j + 128));
                const double2 x0 = *reinterpret_cast<const double2*>(x + j);
                const double2 x1 = *reinterpret_cast<const double2*>(x + j + 2);
                const double2 x2 = *reinterpret_cast<const double2*>(x + j + 128);
                const double2 x3 = *reinterpret_cast<const double2*>(x + j + 130);
                acc0 = fma(widen_f32(a0.x), x0.x, acc0);
                acc1 = fma(widen_f32(a1.x), x2.x, acc1);
                acc0 = fma(widen_f32(a0.y), x0.y, acc0);
                acc1 = fma(widen_f32(a1.y), x2.y, acc1);
                acc0 = fma(widen_f32(a0.z), x1.x, acc0);
                acc1 = fma(widen_f32(a1.z), x3.x, acc1);
                acc0 = fma(widen_f32(a0.w), x1.y, acc0);
                acc1 = fma(widen_f32(a1.w), x3.y, acc1);
            }
            for (; j < n; j += 32 * 4) {
                const float4 a0 = __ldcs(reinterpret_cast<const float4*>(row + j));
                acc0 = fma(widen_f32(a0.x), x[j], acc0);
                acc0 = fma(widen_f32(a0.y), x[j + 1], acc0);
                acc0 = fma(widen_f32(a0.z), x[j + 2], acc0);
                acc0 = fma(widen_f32(a0.w), x[j + 3], acc0);
            }
        } else {
            for (int64_t j = lane; j < n; j += 32) acc0 = fma(wide64(__ldcs(&row[j])), x[j], acc0);
        }
        double acc = msp::warp_sum(acc0 + acc1);
        if (lane == 0) {
            double v = acc + lam * x[i];
            if (b) v = b[i] - v;
            out[i] = v;
            nn += v * v;
        }
    }
    double tot = block_sum(nn, red);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = tot;
        __threadfence();
        unsigned int t = atomicAdd(counter, 1u);
        am_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    double all = sum_parts(part, 1, gridDim.x, red);
    if (threadIdx.x == 0) {
        *counter = 0;
        if (norm2) *norm2 = all;
    }
}

// ---------------------------------------------------------- level 2

// TC: storage type of C and W (T, or BF16 preconditioner data with T = float)
template <typename T, typename TC = T>
struct L2Args {
    int64_t n, s_pad;
    int mode;
    int phase;              // PHASE_ALL, or the part before / after a k_inner launch
    int res_rows;           // rows of C a block keeps in shared memory
    const TC* C;
    const TC* W;
    const T* B;
    const T* Bt;
    T lam_t;
    double tol_rel2;        // level-1 tolerance^2 (MODE_INIT sets ctl->tol2)
    double inner_tol2;
    int max_inner;
    T* x;
    T* r;
    const T* q;
    T* p;                   // direction (packed A pass: the two buffers p, p + p_ld in turn)
    int64_t p_ld;
    T* z;                   // level-1 preconditioned residual (in/out)
    const float* qpart;     // packed A pass: q_i = sum_slot qpart[slot][i] + lam p_i
    int q_slots;
    int n_dq;               // and the block partials of p^T q, n_dq of them in dq
    const double* dq;
    int64_t q_ld;
    T lam;
    CtlBlock* ctl;
    T* part;                // G x s_pad
    T* gvec;                // s_pad
    T* uvec;
    T* tvec;
    T* zvec;
    T* wdvec;
    double* dpart;          // G x 4
    volatile int* prog;     // pinned host words: iterations done, finished (or null)
};

// Per-lane slice of an s_pad row stored as TS: PL elements as PL/W vectors of
// W elements (one vector load each), element index of vector v, component
// e: v*32*W + lane*W + e; values held as T.
template <typename T, int PL, typename TS = T>
struct RowSlice {
    static constexpr int W = StoreW<TS>::W;
    static constexpr int NVEC = PL / W;
    T v[PL];
    __device__ inline void load(const TS* row, int lane) {
#pragma unroll
        for (int k = 0; k < NVEC; ++k) load_vec(row + k * 32 * W + lane * W, v + k * W);
    }
    __device__ inline T dot_smem(const T* s, int lane) const {
        T a = T(0);
#pragma unroll
        for (int k = 0; k < NVEC; ++k)
#pragma unroll
            for (int e = 0; e < W; ++e) a += v[k * W + e] * s[k * 32 * W + lane * W + e];
        return a;
    }
};

// Two neighbouring values of a stored row, widened.
__device__ inline void load_pair(const float* p, float& a, float& b) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    a = v.x;
    b = v.y;
}
__device__ inline void load_pair(const double* p, double& a, double& b) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    a = v.x;
    b = v.y;
}
__device__ inline void load_pair(const __nv_bfloat16* p, float& a, float& b) {
    const uint32_t v = *reinterpret_cast<const uint32_t*>(p);
    a = __uint_as_float(v << 16);
    b = __uint_as_float(v & 0xFFFF0000u);
}

// Layout of the level-2 kernel for a padded sketch size 32 PL.
template <typename T, typename TC, int PL>
struct L2Shape {
    static constexpr int SP = 32 * PL;
    using Cols = msp::L2Columns<SP, kThreads>;
    static constexpr int U = Cols::pairs;
    static constexpr int NG = Cols::groups;         // row groups of the column pass
    static constexpr int KU = Cols::per_thread;
    static constexpr int SCR = NG * SP > kQScratch ? NG * SP : kQScratch;
    // four full vectors, the scratch of the reductions, r and the row results
    static constexpr size_t fixed = ((size_t)4 * SP + SCR + 2 * kRowChunk) * sizeof(T) + 16;
    static constexpr size_t row = (size_t)SP * sizeof(TC);
    // the level-2 iteration by gram_pass: FP32 arithmetic (in FP64 the products bound the
    // passes, not the reads)
    static constexpr bool once = sizeof(T) == 4;
};

// The rows [row0, row0 + nr) of C of one block: the first nres of them in
// shared memory (copied once, when the kernel starts), the others read from L2.
template <typename TC>
struct BlockRows {
    const TC* g;      // row row0 of C
    const TC* s;      // the same rows, resident
    int nr, nres;
};

// acc (a pair of columns per thread) += sum_i coef[i - cb] c_i over the rows
// [cb, ce) of the block; the rows from L2 first (eight loads in flight), then the
// resident ones.
template <typename T, typename TC, int PL>
__device__ __forceinline__ void cols_pass(const BlockRows<TC>& rows, int cb, int ce, const T* coef,
                                          T (&acc)[L2Shape<T, TC, PL>::KU][2]) {
    using S = L2Shape<T, TC, PL>;
    if (!S::Cols::active((int)threadIdx.x)) return;
    const int grp = S::Cols::group((int)threadIdx.x), u0 = S::Cols::first((int)threadIdx.x);
    int i = max(cb, rows.nres) + grp;
    for (; i + 7 * S::NG < ce; i += 8 * S::NG) {
        T c[8][S::KU][2];
#pragma unroll
        for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int k = 0; k < S::KU; ++k) {
                c[q][k][0] = c[q][k][1] = T(0);
                if (S::Cols::has(u0, k))
                    load_pair(rows.g + (int64_t)(i + q * S::NG) * S::SP + 2 * (u0 + k * kThreads), c[q][k][0],
                              c[q][k][1]);
            }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const T f = coef[i + q * S::NG - cb];
#pragma unroll
            for (int k = 0; k < S::KU; ++k) {
                acc[k][0] += f * c[q][k][0];
                acc[k][1] += f * c[q][k][1];
            }
        }
    }
    auto one = [&](const TC* row, T f) {
#pragma unroll
        for (int k = 0; k < S::KU; ++k) {
            if (!S::Cols::has(u0, k)) continue;
            T c0, c1;
            load_pair(row + 2 * (u0 + k * kThreads), c0, c1);
            acc[k][0] += f * c0;
            acc[k][1] += f * c1;
        }
    };
#pragma unroll 4
    for (; i < ce; i += S::NG) one(rows.g + (int64_t)i * S::SP, coef[i - cb]);
    const int se = min(ce, rows.nres);
#pragma unroll 8
    for (i = cb + grp; i < se; i += S::NG) one(rows.s + (int64_t)i * S::SP, coef[i - cb]);
}

// part[b] = the threads' column sums (row groups added through scr, in order)
template <typename T, typename TC, int PL>
__device__ __forceinline__ void cols_store(T (&acc)[L2Shape<T, TC, PL>::KU][2], T* scr, T* part) {
    using S = L2Shape<T, TC, PL>;
    if constexpr (S::NG == 1) {
#pragma unroll
        for (int k = 0; k < S::KU; ++k) {
            const int u = (int)threadIdx.x + k * kThreads;
            if (S::Cols::active((int)threadIdx.x) && S::Cols::has((int)threadIdx.x, k)) {
                part[2 * u] = acc[k][0];
                part[2 * u + 1] = acc[k][1];
            }
        }
    } else {
        const int grp = (int)threadIdx.x / S::U, u = (int)threadIdx.x % S::U;
        if (grp < S::NG) {
            scr[grp * S::SP + 2 * u] = acc[0][0];
            scr[grp * S::SP + 2 * u + 1] = acc[0][1];
        }
        __syncthreads();
        for (int c = threadIdx.x; c < S::SP; c += kThreads) {
            T v = T(0);
#pragma unroll
            for (int g = 0; g < S::NG; ++g) v += scr[g * S::SP + c];
            part[c] = v;
        }
    }
}

// Butterfly reduce-scatter over 2^K lanes' groups: on entry v[0 .. 2^K), on
// exit lane l holds in v[0] the sum over the warp of entry (l >> (5 - K)) of v.
template <int K, typename T>
__device__ __forceinline__ T reduce_scatter(T* v, int lane) {
#pragma unroll
    for (int s = 0; s < K; ++s) {
        const int wd = 16 >> s, half = (1 << K) >> (s + 1);
        const bool upper = (lane & wd) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const T send = upper ? v[i] : v[i + half];
            const T keep = upper ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, wd);
        }
    }
#pragma unroll
    for (int wd = 16 >> K; wd >= 1; wd >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], wd);
    return v[0];
}

// dot[i - cb] = c_i . vec over the rows [cb, ce) of the block (ce - cb <=
// kRowChunk); vec in shared memory. A warp takes every kNW-th row. Up to PL =
// 32 (FP64: 16) its slice of vec stays in registers and it reduces 8 or 16
// rows' partial dots at once; the rows from L2 come first, two in flight up to PL =
// 16 and one beyond (two spilled registers, and what spills goes to L2: next to
// no L1 is left beside the resident rows. An inner step at s = 1024 took 25.4 us at n =
// 8192 with the spills, 23.2 without).
template <typename T, typename TC, int PL>
__device__ __forceinline__ void dots_pass(const BlockRows<TC>& rows, int cb, int ce, const T* vec, T* dot) {
    constexpr int SP = 32 * PL, W = StoreW<TC>::W;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if constexpr (PL <= (sizeof(T) == 4 ? 32 : 16)) {
        T vs[PL];
#pragma unroll
        for (int k = 0; k < PL / W; ++k)
#pragma unroll
            for (int e = 0; e < W; ++e) vs[k * W + e] = vec[k * 32 * W + lane * W + e];
        // this warp's rows in the order they are read: L2 rows, then resident ones
        const int split = min(max(cb, rows.nres), ce);
        const int ng = split + w < ce ? (ce - split - w + kNW - 1) / kNW : 0;
        const int ns = cb + w < split ? (split - cb - w + kNW - 1) / kNW : 0;
        const int cnt = ng + ns;
        auto index = [&](int o) { return o < ng ? split + w + kNW * o : cb + w + kNW * (o - ng); };
        auto ptr = [&](int o) {
            const int i = index(o);
            return o < ng ? rows.g + (int64_t)i * SP : rows.s + (int64_t)i * SP;
        };
        constexpr int KP = PL * sizeof(T) > 80 ? 3 : 4;      // 2^KP partial dots in registers
        for (int o0 = 0; o0 < cnt; o0 += 1 << KP) {
            T part[1 << KP];
#pragma unroll
            for (int t = 0; t < 1 << KP; t += 2) {
                part[t] = T(0);
                part[t + 1] = T(0);
                if (o0 + t < cnt) {
                    RowSlice<T, PL, TC> c0, c1;
                    c0.load(ptr(o0 + t), lane);
                    const bool two = o0 + t + 1 < cnt;
                    if (two && PL <= 16) c1.load(ptr(o0 + t + 1), lane);
#pragma unroll
                    for (int k = 0; k < PL; ++k) part[t] += c0.v[k] * vs[k];
                    if (two) {
                        if (PL > 16) c1.load(ptr(o0 + t + 1), lane);
#pragma unroll
                        for (int k = 0; k < PL; ++k) part[t + 1] += c1.v[k] * vs[k];
                    }
                }
            }
            const T d = reduce_scatter<KP>(part, lane);
            const int o = o0 + (lane >> (5 - KP));
            if ((lane & ((32 >> KP) - 1)) == 0 && o < cnt) dot[index(o) - cb] = d;
        }
    } else {
        for (int i = cb + w; i < ce; i += kNW) {
            RowSlice<T, PL, TC> c;
            c.load(i < rows.nres ? rows.s + (int64_t)i * SP : rows.g + (int64_t)i * SP, lane);
            const T t = msp::warp_sum(c.dot_smem(vec, lane));
            if (lane == 0) dot[i - cb] = t;
        }
    }
}

// How gram_pass cuts a row: HW warps a row, NVH vectors of it a lane, NR rows in
// flight a warp (32 values a lane, 64 KB an SM).
template <typename T, typename TC, int PL>
struct GramShape {
    static constexpr int W = StoreW<TC>::W, NV = PL / W;
    static constexpr int HW = PL > 16 ? 2 : 1, NP = kNW / HW;
    static constexpr int NVH = (NV + HW - 1) / HW;
    static constexpr int NR = NVH * W >= 32 ? 1 : 32 / (NVH * W);
    static constexpr size_t bytes = (size_t)NP * 32 * PL * sizeof(T);
};

// part = sum_i (c_i . vec) c_i over the block's rows, each row read once: HW warps
// take every NP-th row, form its dot and add it from the registers to their own sums
// of their columns, which scr (NP x SP) combines in order. The two warps of a row
// exchange their halves of the dots through xch at a barrier of their own. dots_pass
// and cols_pass in its place read each row that is not resident twice from L2, and at n =
// 32768, s = 1024 (C as large as L2) from memory: a level-2 step took 53 us, with this 44;
// at n = 16384 and s = 2048 71 and 57, s = 1024 27.2 and 27.1. The scratch costs 32 KB
// of resident rows (64 KB at 2048 columns), and where all rows are resident all the same this
// is quicker too, by a block barrier and a second read of shared memory (n = 8192, s = 512:
// 20.6 and 19.6 us).
template <typename T, typename TC, int PL>
__device__ __forceinline__ void gram_pass(const BlockRows<TC>& rows, const T* vec, T* scr, T* xch, T* part) {
    using G = GramShape<T, TC, PL>;
    constexpr int SP = 32 * PL, W = G::W;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, grp = w / G::HW, h = w % G::HW;
    // vector q of this lane: columns at(q) .. + W of the row
    auto has = [&](int q) { return G::NV % G::HW == 0 || G::HW * q + h < G::NV; };
    auto at = [&](int q) { return (G::HW * q + h) * 32 * W + lane * W; };
    T acc[G::NVH * W];
#pragma unroll
    for (int k = 0; k < G::NVH * W; ++k) acc[k] = T(0);
    int turn = 0;
    auto walk = [&](const TC* base, int first, int end) {
#pragma unroll 1
        for (int i = first + grp; i < end; i += G::NR * G::NP) {
            T c[G::NR][G::NVH * W], d[G::NR];
#pragma unroll
            for (int r = 0; r < G::NR; ++r)
#pragma unroll
                for (int q = 0; q < G::NVH; ++q) {
                    if (i + r * G::NP < end && has(q)) {
                        load_vec(base + (int64_t)(i + r * G::NP) * SP + at(q), c[r] + q * W);
                    } else {
#pragma unroll
                        for (int e = 0; e < W; ++e) c[r][q * W + e] = T(0);
                    }
                }
#pragma unroll
            for (int r = 0; r < G::NR; ++r) d[r] = T(0);
#pragma unroll
            for (int q = 0; q < G::NVH; ++q) {
                if (!has(q)) continue;
                T x[W];
                load_vec(vec + at(q), x);
#pragma unroll
                for (int r = 0; r < G::NR; ++r)
#pragma unroll
                    for (int e = 0; e < W; ++e) d[r] += c[r][q * W + e] * x[e];
            }
#pragma unroll
            for (int r = 0; r < G::NR; ++r) d[r] = msp::warp_sum(d[r]);
            if constexpr (G::HW == 2) {
                T* x = xch + (turn * G::NP + grp) * 2 * G::NR;
                if (lane == 0)
#pragma unroll
                    for (int r = 0; r < G::NR; ++r) x[h * G::NR + r] = d[r];
                asm volatile("bar.sync %0, 64;" ::"r"(1 + grp) : "memory");
#pragma unroll
                for (int r = 0; r < G::NR; ++r) d[r] = x[r] + x[G::NR + r];
                turn ^= 1;
            }
#pragma unroll
            for (int r = 0; r < G::NR; ++r)
#pragma unroll
                for (int k = 0; k < G::NVH * W; ++k) acc[k] += d[r] * c[r][k];
        }
    };
    walk(rows.g, rows.nres, rows.nr);
    walk(rows.s, 0, rows.nres);
#pragma unroll
    for (int q = 0; q < G::NVH; ++q)
        if (has(q))
#pragma unroll
            for (int e = 0; e < W; ++e) scr[grp * SP + at(q) + e] = acc[q * W + e];
    __syncthreads();
    for (int c = threadIdx.x; c < SP; c += kThreads) {
        T v = T(0);
#pragma unroll
        for (int q = 0; q < G::NP; ++q) v += scr[q * SP + c];
        part[c] = v;
    }
}

// out[c] = M[c,:] . svec for c in [c0, c1) (warp per row)
template <typename T, int PL, typename TS = T>
__device__ inline void rows_dot(const TS* M, int64_t s_pad, int64_t c0, int64_t c1, const T* svec,
                                T* out) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t c = c0 + w; c < c1; c += kNW) {
        RowSlice<T, PL, TS> m;
        m.load(M + c * s_pad, lane);
        T t = msp::warp_sum(m.dot_smem(svec, lane));
        if (lane == 0) out[c] = t;
    }
}

// out[c] = sum_k part[k][c] (+ add_scale * addend[c]) over the block's columns,
// the groups of eight b, b + G, ...; k < G <= kThreads. Thread k reads the eight
// columns of partial k (one or two sectors), a warp reduces them by a
// reduce-scatter, and threads c < 8 add the warps' sums in order in FP64. With
// dvec (shared memory) returns sum_c dvec[c] out[c], with sq sum_c out[c]^2, in
// thread 0. red holds kNW x 8 values. Ends past a block barrier.
template <typename T>
__device__ inline double reduce_cols(const T* part, int G, int64_t sp, const T* addend, T add_scale, T* out,
                                     const T* dvec, bool sq, T* red) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (G + 31) >> 5;
    constexpr int W = Vec16<T>::W;
    double dot = 0.0;
    int64_t cb = (int64_t)blockIdx.x * 8;
    do {
        if (w < nw && cb < sp) {
            T v[8];
            const T* row = part + (int64_t)threadIdx.x * sp + cb;
#pragma unroll
            for (int k = 0; k < 8; k += W) {
                if ((int)threadIdx.x < G) {
                    const typename Vec16<T>::type q =
                        __ldcg(reinterpret_cast<const typename Vec16<T>::type*>(row + k));
                    if constexpr (W == 4) { v[k] = q.x; v[k + 1] = q.y; v[k + 2] = q.z; v[k + 3] = q.w; }
                    else { v[k] = q.x; v[k + 1] = q.y; }
                } else {
#pragma unroll
                    for (int e = 0; e < W; ++e) v[k + e] = T(0);
                }
            }
            const T t = reduce_scatter<3>(v, lane);
            if ((lane & 3) == 0) red[w * 8 + (lane >> 2)] = t;
        }
        __syncthreads();
        if (threadIdx.x < 8 && cb < sp) {
            const int64_t c = cb + threadIdx.x;
            double acc = 0.0;
            for (int k = 0; k < nw; ++k) acc += (double)red[k * 8 + threadIdx.x];
            T r = (T)acc;
            if (addend) r += add_scale * __ldcg(&addend[c]);
            out[c] = r;
            if (dvec) dot += (double)dvec[c] * (double)r;
            else if (sq) dot += (double)r * (double)r;
        }
        cb += 8 * (int64_t)G;
        if (cb < sp) __syncthreads();
    } while (cb < sp);
    if ((dvec || sq) && w == 0)
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    return dot;
}

// Sum over the block in warp 0; `active`: this warp holds values (the same in
// all its lanes; a warp without any adds nothing to the FP64 pipe). red: kNW.
__device__ inline double block_sum0(double v, bool active, double* red) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (active) v = msp::warp_sum(v);
    if (lane == 0) red[w] = active ? v : 0.0;
    __syncthreads();
    if (w != 0) return 0.0;
    return msp::warp_sum(lane < kNW ? red[lane] : 0.0);
}

// Sum of a per-block partial array by the calling warp, fixed order.
__device__ inline double warp_sum_parts(const double* parts, int stride, int G) {
    double v = 0.0;
    for (int k = threadIdx.x & 31; k < G; k += 32) v += __ldcg(&parts[(int64_t)k * stride]);
    return msp::warp_sum(v);
}

// The same for every thread: warp 0 sums, *slot hands the value on. A slot is
// written again only after a later block barrier.
__device__ inline double grid_sum(const double* parts, int G, double* slot) {
    if ((threadIdx.x >> 5) == 0) {
        const double v = warp_sum_parts(parts, 4, G);
        if (threadIdx.x == 0) *slot = v;
    }
    __syncthreads();
    return *slot;
}

template <typename T>
__device__ inline void load_full(const T* g, T* s, int64_t m) {
    for (int64_t c = threadIdx.x; c < m; c += blockDim.x) s[c] = __ldcg(&g[c]);
}

// One block of 16 warps per SM. What bounds it is latency: the grid barriers
// and the serial phases between them; after those, the FP64 pipe (2 lanes a clock
// an SM, a warp-wide FP64 instruction holds it for 16 cycles), so every FP64 sum
// is formed by the warps that hold values and finished by one warp, and the two
// passes over the block's rows of C. The first res_rows of those rows are copied
// to shared memory by the copy engine when the kernel starts, beside the level-1
// update, and serve every pass (at n = 8192, s = 512 all of them; at n = 16384,
// s = 1024 a third). Two blocks of 8 warps per SM, every warp finishing every sum,
// the rows read twice from L2, and the new direction formed here behind a fifth
// barrier took 36.6 us (n = 16384, s = 1024) and 28.5 us (n = 8192, s = 512); now
// 27.8 and 20.5 us.
template <typename T, typename TC, int PL>
__global__ void __launch_bounds__(kThreads, 1) k_level2(L2Args<T, TC> a) {
    using S = L2Shape<T, TC, PL>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int64_t sp = S::SP;
    TC* cres = reinterpret_cast<TC*>(smem_raw);   // resident rows of C
    T* sd = reinterpret_cast<T*>(smem_raw + (size_t)a.res_rows * S::row);   // d (search direction)
    T* sres = sd + sp;                            // level-2 residual
    T* sy = sres + sp;                            // level-2 iterate
    T* stmp = sy + sp;                            // scratch full vector
    T* scr = stmp + sp;                           // reduction scratch
    T* srow = scr + S::SCR;                       // r of the block's rows (a chunk)
    T* sw = srow + kRowChunk;                     // row results
    uint64_t* bar = reinterpret_cast<uint64_t*>(sw + kRowChunk);
    __shared__ double red[kNW], red_b[kNW], red_c[kNW];
    __shared__ T redc[kNW * 8];
    __shared__ double s_alpha, s_rr, s_val[4];
    __shared__ int s_bad, s_stop;

    CtlBlock* ctl = a.ctl;
    // the control words in one round trip
    const int c_done = ctl->done, c_err = ctl->error, iter = ctl->iters;
    const double c_alpha = ctl->alpha, c_rz = ctl->rz, tol2 = ctl->tol2;
    const double c_rz0 = ctl->rzbuf[0], c_rz1 = ctl->rzbuf[1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int G = gridDim.x, b = blockIdx.x;
    // tells the host that polls for it (block 0)
    auto report = [&](int word, int v) {
        if (a.prog && b == 0 && threadIdx.x == 0) a.prog[word] = v;
    };
    const int64_t row0 = a.n * b / G, row1 = a.n * (b + 1) / G;
    const int64_t c0 = sp * b / G, c1 = sp * (b + 1) / G;
    unsigned int* bw = &ctl->bar_word;
    int* err = &ctl->error;
    const bool packed = a.dq != nullptr;
    BlockRows<TC> rows{a.C + row0 * sp, cres, (int)(row1 - row0), (int)min((int64_t)a.res_rows, row1 - row0)};
    // thread 0's view of the flags stands for its block: block 0 may store an error
    // (s_bad below) while other blocks are still starting, and a block leaves whole or
    // not at all
    if (threadIdx.x == 0) s_stop = c_done | c_err;
    if (threadIdx.x == 0 && !(c_done | c_err)) {
        msp::mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        uint32_t left = (uint32_t)(rows.nres * S::row);
        msp::mbar_arrive_expect_tx(bar, left);
        for (uint32_t o = 0; left > 0;) {
            const uint32_t len = min(left, 32768u);
            msp::bulk_g2s(smem_raw + o, reinterpret_cast<const unsigned char*>(rows.g) + o, len, bar);
            o += len;
            left -= len;
        }
        s_bad = 0;
    }
    __syncthreads();
    if (s_stop) {
        report(1, 1);
        return;
    }

    // ---- level-1 update
    const T* p = a.p;
    bool have_r = false;      // srow holds r of all the block's rows
    double rr = 0.0;
    if (a.phase == PHASE_BACK) {
    } else if (a.mode == MODE_ITER && packed) {
        // q_i = sum over the packed A pass's slot partials + lam p_i, fixed
        // summation order. Rounds of four 32-row groups: every warp sums its
        // slots for the four rows of a lane, the loads in flight together
        // (eight slots per row at a time), warp g finishes group g (its p_i,
        // r_i, x_i loaded before the slot partials). The last warp takes no
        // slots: it forms the step alpha = rz / p^T q meanwhile.
        constexpr int kGroups = 4;
        p = a.p + (iter & 1) * a.p_ld;
        T* sq = scr;          // kGroups x kNS x 32
        constexpr int kNS = kNW - 1;
        if (w == kNW - 1) {
            const double pq = warp_sum_parts(a.dq, 1, a.n_dq);
            if (lane == 0) {
                s_alpha = ((iter & 1) ? c_rz1 : c_rz0) / pq;
                if (!isfinite(pq)) s_bad = MSP_ENONFINITE;
                else if (!(pq > 0.0)) s_bad = MSP_ENOTPD;
            }
        }
        // p^T q not positive or not finite: block 0 records it, and every block leaves (the
        // sum and so the outcome are the same in all of them). Called past a block barrier.
        auto breakdown = [&]() -> bool {
            if (!s_bad) return false;
            if (threadIdx.x == 0) {
                if (b == 0) atomicExch(err, s_bad);
                msp::mbar_wait_timed(bar, 0, err);   // the resident rows land before the block leaves
            }
            return true;
        };
        have_r = rows.nr <= kRowChunk;
        if (rows.nr == 0) {       // fewer rows than blocks
            __syncthreads();
            if (breakdown()) return;
        }
        for (int64_t base = row0; base < row1; base += 32 * kGroups) {
            const int64_t i_own = base + 32 * w + lane;      // the row this thread finishes (w < kGroups)
            const bool own = w < kGroups && i_own < row1;
            T p_own = T(0), r_own = T(0), x_own = T(0);
            if (own) {
                p_own = p[i_own];
                r_own = a.r[i_own];
                x_own = a.x[i_own];
            }
            T v[kGroups];
#pragma unroll
            for (int g = 0; g < kGroups; ++g) v[g] = T(0);
            int sl = w < kNS ? w : a.q_slots;
            for (; sl + 7 * kNS < a.q_slots; sl += 8 * kNS) {
                T t8[kGroups][8];
#pragma unroll
                for (int g = 0; g < kGroups; ++g) {
                    const int64_t i = base + 32 * g + lane;
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        t8[g][u] = (i < row1) ? __ldcg(&a.qpart[(int64_t)(sl + u * kNS) * a.q_ld + i]) : T(0);
                }
#pragma unroll
                for (int g = 0; g < kGroups; ++g)
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[g] += t8[g][u];
            }
            for (; sl < a.q_slots; sl += 2 * kNS) {
                const bool two = sl + kNS < a.q_slots;
                T t0[kGroups], t1[kGroups];
#pragma unroll
                for (int g = 0; g < kGroups; ++g) {
                    const int64_t i = base + 32 * g + lane;
                    t0[g] = (i < row1) ? __ldcg(&a.qpart[(int64_t)sl * a.q_ld + i]) : T(0);
                    t1[g] = (two && i < row1) ? __ldcg(&a.qpart[(int64_t)(sl + kNS) * a.q_ld + i]) : T(0);
                }
#pragma unroll
                for (int g = 0; g < kGroups; ++g) v[g] = (v[g] + t0[g]) + t1[g];
            }
#pragma unroll
            for (int g = 0; g < kGroups; ++g)
                if (w < kNS) sq[(g * kNS + w) * 32 + lane] = v[g];
            __syncthreads();
            if (breakdown()) return;
            if (own) {
                const T alpha = (T)s_alpha;
                T qi = T(0);
#pragma unroll
                for (int g = 0; g < kNS; ++g) qi += sq[(w * kNS + g) * 32 + lane];
                qi += a.lam * p_own;
                T ri = r_own;
                a.x[i_own] = x_own + alpha * p_own;
                ri -= alpha * qi;
                a.r[i_own] = ri;
                if (have_r) srow[i_own - row0] = ri;
                rr += (double)ri * (double)ri;
            }
            __syncthreads();
        }
        rr = block_sum0(rr, w < kGroups, red);
    } else if (a.mode != MODE_APPLY) {
        for (int64_t i = row0 + threadIdx.x; i < row1; i += blockDim.x) {
            T ri = a.r[i];
            if (a.mode == MODE_ITER) {
                const T alpha = (T)c_alpha;
                a.x[i] += alpha * p[i];
                ri -= alpha * a.q[i];
                a.r[i] = ri;
            }
            rr += (double)ri * (double)ri;
        }
        rr = block_sum0(rr, 32 * w < rows.nr, red);
    }
    if (threadIdx.x == 0 && a.phase != PHASE_BACK) a.dpart[b * 4 + 0] = rr;

    // the block's rows of r (a chunk) in srow
    auto load_r = [&](int cb, int ce) {
        for (int e = cb + (int)threadIdx.x; e < ce; e += kThreads) srow[e - cb] = a.r[row0 + e];
        __syncthreads();
    };
    // ---- g = C^T r partials. A copy that does not arrive is seen by every thread
    // that waits for it; the block then leaves and the others' grid barrier runs out.
    T acc[S::KU][2];
#pragma unroll
    for (int k = 0; k < S::KU; ++k) acc[k][0] = acc[k][1] = T(0);
    if (!msp::mbar_wait_timed(bar, 0, err)) s_bad = MSP_ETIMEOUT;
    int k = 0;                // level-2 iterations
    if (a.phase != PHASE_BACK) {
        for (int cb = 0; cb < rows.nr; cb += kRowChunk) {
            const int ce = min(rows.nr, cb + kRowChunk);
            if (!have_r) load_r(cb, ce);
            cols_pass<T, TC, PL>(rows, cb, ce, srow, acc);
            if (ce < rows.nr) __syncthreads();
        }
        have_r = rows.nr <= kRowChunk;   // srow is not written again below
        cols_store<T, TC, PL>(acc, scr, a.part + (int64_t)b * sp);
        // the block's rows of B and B^T on their way to registers during the barriers
        // (PL > 32: two rows of that length would not fit the registers)
        const bool one_row = PL <= 32 && c1 - c0 <= kNW;
        const bool my_row = one_row && c0 + w < c1 && a.phase == PHASE_ALL;
        RowSlice<T, PL> mB;
        if (my_row) mB.load(a.B + (c0 + w) * sp, lane);
        if (!msp::grid_barrier(bw, err) || s_bad) return;

        // ---- g reduced over this block's columns, |r|^2 (the convergence test) by
        // the last warp beside it; |g|^2 only where the level-2 iteration's tolerance needs it
        const bool inner = a.max_inner > 0 && a.phase == PHASE_ALL;
        if (a.mode != MODE_APPLY && w == kNW - 1) {
            const double t = warp_sum_parts(a.dpart, 4, G);
            if (lane == 0) s_rr = t;
        }
        double gg = reduce_cols<T>(a.part, G, sp, nullptr, T(0), a.gvec, nullptr, inner, redc);
        if (a.mode != MODE_APPLY) {
            rr = s_rr;
            bool stop = !isfinite(rr);
            double t2 = tol2;
            if (a.mode == MODE_INIT) t2 = a.tol_rel2 * rr;
            if (stop) {
                if (b == 0 && threadIdx.x == 0) ctl->error = MSP_ENONFINITE;
                return;
            }
            if (rr <= t2) {
                if (b == 0 && threadIdx.x == 0) {
                    ctl->rr = rr;
                    if (a.mode == MODE_INIT) { ctl->bb = rr; ctl->tol2 = t2; }
                    if (a.mode == MODE_ITER) ctl->iters = iter + 1;
                    ctl->done = 1;
                }
                return;
            }
        }
        if (a.mode != MODE_APPLY && b == 0 && threadIdx.x == 0) {
            ctl->rr = rr;
            if (a.mode == MODE_INIT) { ctl->bb = rr; ctl->tol2 = a.tol_rel2 * rr; }
        }
        if (a.phase == PHASE_FRONT) return;
        if (inner && threadIdx.x == 0) a.dpart[b * 4 + 1] = gg;
        if (!msp::grid_barrier(bw, err)) return;
        if (inner) gg = grid_sum(a.dpart + 1, G, &s_val[0]);
        load_full(a.gvec, sres, sp);
        if (inner)
            for (int c = threadIdx.x; c < sp; c += kThreads) sy[c] = T(0);
        __syncthreads();

        // ---- z = M2^{-1} res = B^T (B res); z^T res only where the level-2
        // iteration uses it (rz_out given; the same in every block)
        int turn = 1;
        bool fresh = my_row;      // mB holds the block's row of B
        auto precond = [&](double* rz_out) -> bool {
            RowSlice<T, PL> mT;
            if (my_row) {
                if (!fresh) mB.load(a.B + (c0 + w) * sp, lane);
                fresh = false;
                const T t = msp::warp_sum(mB.dot_smem(sres, lane));
                if (lane == 0) a.tvec[c0 + w] = t;
                mT.load(a.Bt + (c0 + w) * sp, lane);
            } else if (!one_row) {
                rows_dot<T, PL>(a.B, sp, c0, c1, sres, a.tvec);
            }
            if (!msp::grid_barrier(bw, err)) return false;
            load_full(a.tvec, stmp, sp);
            __syncthreads();
            double part = 0.0;
            if (my_row) {
                const T z = msp::warp_sum(mT.dot_smem(stmp, lane));
                if (lane == 0) {
                    a.zvec[c0 + w] = z;
                    if (rz_out) part = (double)sres[c0 + w] * (double)z;
                }
            } else if (!one_row) {
                rows_dot<T, PL>(a.Bt, sp, c0, c1, stmp, a.zvec);
                __syncthreads();
                if (rz_out)
                    for (int64_t c = c0 + threadIdx.x; c < c1; c += kThreads) part += (double)sres[c] * (double)a.zvec[c];
            }
            if (rz_out) {
                // my_row: lane 0 of each warp holds a product
                if (one_row) {
                    if (lane == 0) red_b[w] = part;
                    __syncthreads();
                    part = w == 0 ? msp::warp_sum(lane < kNW ? red_b[lane] : 0.0) : 0.0;
                } else {
                    part = block_sum0(part, true, red_b);
                }
                if (threadIdx.x == 0) a.dpart[b * 4 + 2] = part;
            }
            if (!msp::grid_barrier(bw, err)) return false;
            if (rz_out) {
                *rz_out = grid_sum(a.dpart + 2, G, &s_val[turn]);
                turn = 3 - turn;
            }
            return true;
        };

        // direct level 2 (max_inner == 0) has no level-2 iteration: z^T res unused
        double rz_in = 0.0;
        if (!precond(inner ? &rz_in : nullptr)) return;
        // direct level 2: M2 is the level-2 operator itself (Phi = I), so
        // y = M2^{-1} C^T r with no correction steps
        load_full(a.zvec, inner ? sd : sy, sp);
        __syncthreads();
        double rres = gg;
        const double tin2 = a.inner_tol2 * gg;
        while (k < a.max_inner && rres > tin2) {
            // P1: partial u = C^T (C d) over this block's rows; wd = W d (columns)
            if constexpr (S::once) {
                T* wscr = reinterpret_cast<T*>(smem_raw + (size_t)a.res_rows * S::row + S::fixed);
                gram_pass<T, TC, PL>(rows, sd, wscr, sw, a.part + (int64_t)b * sp);
            } else {
#pragma unroll
                for (int q = 0; q < S::KU; ++q) acc[q][0] = acc[q][1] = T(0);
                for (int cb = 0; cb < rows.nr; cb += kRowChunk) {
                    const int ce = min(rows.nr, cb + kRowChunk);
                    dots_pass<T, TC, PL>(rows, cb, ce, sd, sw);
                    __syncthreads();
                    cols_pass<T, TC, PL>(rows, cb, ce, sw, acc);
                    if (ce < rows.nr) __syncthreads();
                }
                cols_store<T, TC, PL>(acc, scr, a.part + (int64_t)b * sp);
            }
            rows_dot<T, PL, TC>(a.W, sp, c0, c1, sd, a.wdvec);
            if (!msp::grid_barrier(bw, err)) return;
            // P2: u over this block's columns; d.u partial
            double du = reduce_cols<T>(a.part, G, sp, a.wdvec, a.lam_t, a.uvec, sd, false, redc);
            if (threadIdx.x == 0) a.dpart[b * 4 + 3] = du;
            if (!msp::grid_barrier(bw, err)) return;
            // P3: step
            du = grid_sum(a.dpart + 3, G, &s_val[3]);
            if (!(du > 0.0)) break;   // breakdown (same decision in every block)
            const T ain = (T)(rz_in / du);
            double loc = 0.0;
            for (int c = threadIdx.x; c < sp; c += kThreads) {
                T u = __ldcg(&a.uvec[c]);
                sy[c] += ain * sd[c];
                T rv = sres[c] - ain * u;
                sres[c] = rv;
                loc += (double)rv * (double)rv;
            }
            rres = block_sum0(loc, 32 * w < sp, red_c);
            if (threadIdx.x == 0) s_val[0] = rres;
            __syncthreads();
            rres = s_val[0];
            ++k;
            if (rres <= tin2) break;
            double rz_new = 0.0;
            if (!precond(&rz_new)) return;
            const T beta = (T)(rz_new / rz_in);
            rz_in = rz_new;
            for (int c = threadIdx.x; c < sp; c += kThreads) sd[c] = __ldcg(&a.zvec[c]) + beta * sd[c];
            __syncthreads();
        }
    } else {
        if (s_bad) return;
        load_full(a.zvec, sy, sp);     // y of the k_inner launch
    }

    // ---- w = (r - C y) / lam~ into z; dots r.w and r.z_old for the level-1 beta
    __syncthreads();
    double rw = 0.0, rzo = 0.0;
    for (int cb = 0; cb < rows.nr; cb += kRowChunk) {
        const int ce = min(rows.nr, cb + kRowChunk);
        if (!have_r) load_r(cb, ce);
        T zo = T(0);
        const int e = cb + (int)threadIdx.x;      // kRowChunk = kThreads: a row per thread
        if (a.mode == MODE_ITER && e < ce) zo = a.z[row0 + e];
        dots_pass<T, TC, PL>(rows, cb, ce, sy, sw);
        __syncthreads();
        if (e < ce) {
            const T ri = srow[e - cb], wi = (ri - sw[e - cb]) / a.lam_t;
            a.z[row0 + e] = wi;
            if (a.mode != MODE_APPLY) {
                rw += (double)ri * (double)wi;
                rzo += (double)ri * (double)zo;
            }
        }
        if (ce < rows.nr) __syncthreads();
    }
    if (a.mode == MODE_APPLY) {
        if (b == 0 && threadIdx.x == 0) ctl->inner_iters += k;
        return;
    }
    {
        // rw by the warps that have rows, finished by warp 0; rzo by warp 1
        if (32 * w < rows.nr) {
            rw = msp::warp_sum(rw);
            if (a.mode == MODE_ITER) rzo = msp::warp_sum(rzo);
        }
        if (lane == 0) {
            red_b[w] = rw;
            red_c[w] = rzo;
        }
        __syncthreads();
        if (w < 2) {
            const double t = msp::warp_sum(lane < kNW ? (w == 0 ? red_b[lane] : red_c[lane]) : 0.0);
            if (lane == 0) a.dpart[b * 4 + w] = t;
        }
    }
    // packed A pass: the next launch (the A pass) is the barrier; it sums the
    // partials, checks r^T w and forms beta and the new direction
    if (!packed) {
        if (!msp::grid_barrier(bw, err)) return;
        if (w < 2) {
            const double t = warp_sum_parts(a.dpart + w, 4, G);
            if (lane == 0) s_val[w] = t;
        }
        __syncthreads();
        rw = s_val[0];
        rzo = s_val[1];
        T beta = T(0);
        if (a.mode == MODE_ITER) beta = (T)((rw - rzo) / c_rz);
        for (int64_t i = row0 + threadIdx.x; i < row1; i += kThreads)
            a.p[i] = a.z[i] + beta * (a.mode == MODE_ITER ? a.p[i] : T(0));
        if (b == 0 && threadIdx.x == 0) {
            ctl->rz = rw;
            ctl->beta = (double)beta;
            if (!(rw > 0.0) && isfinite(rw)) ctl->error = MSP_ENOTPD;
            if (!isfinite(rw)) ctl->error = MSP_ENONFINITE;
        }
    }
    if (b == 0 && threadIdx.x == 0) {
        ctl->inner_iters += k;
        if (a.mode == MODE_ITER) {
            ctl->iters = iter + 1;
            report(0, iter + 1);
        }
    }
}

template <typename T, typename TC, int PL>
msp_status launch_level2_pl(msp_ctx* ctx, L2Args<T, TC>& a, int G) {
    using S = L2Shape<T, TC, PL>;
    auto kern = k_level2<T, TC, PL>;
    // rows of C kept in shared memory: what the block's rows need, or what is
    // left beside the vectors (4 KB aside for the kernel's static part)
    const size_t left = ctx->smem_optin - 4096 - S::fixed;
    const int64_t most = (a.n + G - 1) / G;
    size_t scratch = 0;       // gram_pass's, behind the vectors
    if constexpr (S::once)
        if (a.max_inner > 0 && a.phase == PHASE_ALL) scratch = GramShape<T, TC, PL>::bytes;
    const int64_t fit = (int64_t)((left - scratch) / S::row);
    a.res_rows = (int)(fit >= most ? most : scratch ? fit : fit / kNW * kNW);
    const size_t smem = S::fixed + (size_t)a.res_rows * S::row + scratch;
    MSP_CUDA_TRY(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)smem));
    // co-residency is required by the grid barrier: never exceed what fits
    int per_sm = 0;
    MSP_CUDA_TRY(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem));
    if (per_sm < 1)
        return msp_set_error(ctx, MSP_EINVAL, "level-2 kernel does not fit on an SM");
    void* args[] = {&a};
    ++ctx->launches;
    MSP_CUDA_TRY(ctx, cudaLaunchCooperativeKernel((const void*)kern, dim3(G), dim3(kThreads), args,
                                                  smem, ctx->stream));
    return MSP_OK;
}

template <typename T, typename TC>
msp_status launch_level2(msp_ctx* ctx, L2Args<T, TC>& a, int G) {
    // one instantiation per padded sketch size (multiples of 128 up to 1024,
    // then 1536 and 2048)
    switch (a.s_pad) {
        case 128: return launch_level2_pl<T, TC, 4>(ctx, a, G);
        case 256: return launch_level2_pl<T, TC, 8>(ctx, a, G);
        case 384: return launch_level2_pl<T, TC, 12>(ctx, a, G);
        case 512: return launch_level2_pl<T, TC, 16>(ctx, a, G);
        case 640: return launch_level2_pl<T, TC, 20>(ctx, a, G);
        case 768: return launch_level2_pl<T, TC, 24>(ctx, a, G);
        case 896: return launch_level2_pl<T, TC, 28>(ctx, a, G);
        case 1024: return launch_level2_pl<T, TC, 32>(ctx, a, G);
        case 1536:
            if constexpr (sizeof(T) == 4) return launch_level2_pl<T, TC, 48>(ctx, a, G);
            break;
        case 2048:
            if constexpr (sizeof(T) == 4) return launch_level2_pl<T, TC, 64>(ctx, a, G);
            break;
        default: break;
    }
    return msp_set_error(ctx, MSP_EINVAL, "level-2: unsupported padded sketch size %lld",
                         (long long)a.s_pad);
}

// ------------------------------------------------ level-2 iteration on a formed operator

template <typename T>
struct InnerArgs {
    const T* H;             // C^T C + lam~ W, s_pad x s_pad (FP32: rounded), null: not formed
    const float* Hlo;       // FP32: what the rounding left
    const T* B;
    const T* Bt;
    const T* g;             // C^T r
    T* y;
    double inner_tol2;
    int max_inner;
    CtlBlock* ctl;
};

// The level-2 PCG of Algorithm 2 on (C^T C + lam~ W) y = g, preconditioned by
// M2^{-1} v = B^T (B v), as products with the formed s_pad x s_pad operator, on one
// cluster of 16 CTAs. In k_level2 an iteration is a pass over C and four grid
// barriers (18 us at n = 4999, s = 312; 18 us in FP64 at n = 1024, s = 64); here it is
// three products on data that stays on the SMs, with an exchange each: 5.1 us
// and 5.0 us.
//
// A CTA has s_pad / 16 rows of H, B and B^T, 16 lanes a row, E = s_pad / 16 values of
// a row a lane, in registers for the whole launch (at s_pad = 384 in FP32, H a pair, 60
// bytes of them spill). The row sums are gathered
// in shared memory and sent to every CTA's copy of the result by 16-byte st.async
// pieces that count on that CTA's mbarrier (two copies in turn: a CTA sends product
// k + 2 only after it has every CTA's part of k + 1, sent after the reads of k);
// thread t of every CTA has component t. What bounds it is the latency of that
// chain, so the dots and quotients, formed in every CTA from the same values in
// the same order, belong to four more warps (one per FP64 unit: a warp-wide FP64
// sum takes 520 cycles, a quotient 560 in one warp and 1540 in four), and
// |res|^2 is taken while the product with B that follows it is under way. One thread
// polls the mbarrier and the others wait at the block barrier: with a cluster
// barrier instead, the waiting warps' polls slowed the others' shuffles (a
// FP64 sum 2700 cycles, four FP32 steps 950) and an iteration took 6 us. FP32: H as a
// pair of floats, so the operator is that of the compensated Gram, not its rounding.
constexpr int kInnerCtas = 16;
constexpr int kDotThreads = 128;

// Exact widening without the FP64 pipe for normal numbers.
__device__ __forceinline__ double widen_exact(double v) { return v; }
__device__ __forceinline__ double widen_exact(float x) {
    const uint32_t b = __float_as_uint(x);
    if (((b >> 23) & 0xFFu) - 1u >= 254u) return (double)x;     // zero, subnormal, infinity, NaN
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20))), (int)(b << 29));
}

// 16 bytes of this CTA's shared memory to the same place as `dst` in CTA `to` of the
// cluster, counted on that CTA's `bar`
template <typename T>
__device__ __forceinline__ void st_async16(T* dst, const T* src, uint64_t* bar, int to) {
    uint32_t d, b;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(msp::smem_u32(dst)), "r"(to));
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(msp::smem_u32(bar)), "r"(to));
    const uint4 v = *reinterpret_cast<const uint4*>(src);
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(d),
                 "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(b)
                 : "memory");
}

template <typename T, int E>
__global__ void __launch_bounds__(16 * E + kDotThreads, 1) k_inner(InnerArgs<T> a) {
    namespace cg = cooperative_groups;
    constexpr int SP = 16 * E, OWN = SP / kInnerCtas, W = Vec16<T>::W, NV = E / W;
    constexpr int VPD = OWN / W;              // 16-byte pieces of a CTA's rows
    static_assert(VPD * kInnerCtas <= SP, "a piece per thread");
    cg::cluster_group cl = cg::this_cluster();
    __shared__ __align__(16) T va[SP], vb[SP], ybuf[2][SP], stage[OWN];
    __shared__ __align__(8) uint64_t full[2];
    __shared__ double red[4], s_sc, s_rres;
    __shared__ int s_bad;
    CtlBlock* ctl = a.ctl;
    if (ctl->done | ctl->error) return;       // the same in every CTA: nothing writes them here
    const int tid = threadIdx.x, lane = tid & 31, l16 = tid & 15;
    const bool dots = tid >= SP;              // the warps of the dots
    const int rank = (int)cl.block_rank();
    const int row = rank * OWN + (tid >> 4);
    constexpr int NP = sizeof(T) == 4 ? 2 : 1;
    T h[E], hl[NP == 2 ? E : 1], bm[E], bt[E];
    T res = T(0), y = T(0), d = T(0);
    if (!dots) {
        auto load_row = [&](const T* M, T* dst) {
#pragma unroll
            for (int k = 0; k < NV; ++k) load16(M + (int64_t)row * SP + W * (l16 + 16 * k), dst + k * W);
        };
        load_row(a.B, bm);
        load_row(a.Bt, bt);
        load_row(a.H, h);
        if constexpr (NP == 2) load_row(a.Hlo, hl);
        res = a.g[tid];
        va[tid] = res;
    }
    if (tid == 0) {
        msp::mbar_init(&full[0], 1);
        msp::mbar_init(&full[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_bad = 0;
    }
    cl.sync();   // every CTA runs, its mbarriers ready, before it is written to
    uint32_t sent = 0;                        // products so far
    // u . v (shared memory) in the first of the dots' warps
    auto dot = [&](const T* u, const T* v) -> double {
        double t = 0.0;
#pragma unroll
        for (int c = tid - SP; c < SP; c += kDotThreads) t = fma(widen_exact(u[c]), widen_exact(v[c]), t);
        t = msp::warp_sum(t);
        if (lane == 0) red[(tid - SP) >> 5] = t;
        asm volatile("bar.sync 2, %0;" ::"n"(kDotThreads) : "memory");
        return (red[0] + red[1]) + (red[2] + red[3]);
    };
    // f(u . v) for every thread; ends past a block barrier
    auto scalar = [&](const T* u, const T* v, auto f) -> double {
        if (dots) {
            const double t = dot(u, v);
            if (tid < SP + 32) {
                const double q = f(t);
                if (lane == 0) s_sc = q;
            }
        }
        __syncthreads();
        return s_sc;
    };
    // M v, v in shared memory (visible to the block): the copy of the full
    // result. with_rr: |v|^2 into s_rres meanwhile. Ends past a block barrier.
    auto product = [&](const T* m, const T* mlo, const T* v, bool with_rr) -> const T* {
        if (!dots) {
            T s0 = T(0), s1 = T(0);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                T x[W];
                load16(v + W * (l16 + 16 * k), x);
#pragma unroll
                for (int e = 0; e < W; ++e) {
                    s0 = fma(m[k * W + e], x[e], s0);
                    if (mlo) s1 = fma(mlo[k * W + e], x[e], s1);
                }
            }
            s0 += s1;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
            if (l16 == 0) stage[tid >> 4] = s0;
            asm volatile("bar.sync 1, %0;" ::"n"(SP) : "memory");
            if (tid < VPD * kInnerCtas) {
                const int to = tid / VPD, piece = tid % VPD;
                st_async16(&ybuf[sent & 1][rank * OWN + piece * W], stage + piece * W, &full[sent & 1], to);
            }
            // a phase whose wait ran out takes no second arrival: this CTA waits no more, and
            // leaves at the next test of s_bad
            if (tid == 0 && !s_bad) {
                msp::mbar_arrive_expect_tx(&full[sent & 1], SP * (uint32_t)sizeof(T));
                if (!msp::mbar_wait_timed<true>(&full[sent & 1], (sent >> 1) & 1u, &ctl->error)) s_bad = 1;
            }
        } else if (with_rr) {
            const double t = dot(v, v);
            if (tid == SP) s_rres = t;
        }
        __syncthreads();
        return ybuf[sent++ & 1];
    };
    const T* z = nullptr;
    double rz = 0.0;             // r^T z, in the dots' first warp
    int k = 0;
    // t = B res (res in va) and |res|^2; with t in vb, z = B^T t
    auto half = [&]() {
        const T* t = product(bm, nullptr, va, true);
        if (!dots) vb[tid] = t[tid];
        __syncthreads();
        return s_rres;
    };
    const double gg = half(), tin2 = a.inner_tol2 * gg;
    if (gg > tin2 && a.max_inner > 0 && !s_bad) {
        z = product(bt, nullptr, vb, false);
        scalar(va, z, [&](double t) { return rz = t; });
        if (!dots) d = z[tid];
        while (true) {
            if (!dots) vb[tid] = d;
            __syncthreads();
            const T* u = product(h, NP == 2 ? hl : nullptr, vb, false);
            // the step, NaN for a breakdown (d . u not positive)
            const double q = scalar(vb, u, [&](double du) { return du > 0.0 ? rz / du : nan(""); });
            if (!(q == q)) break;
            if (!dots) {
                const T ain = (T)q;
                y += ain * d;
                res -= ain * u[tid];
                va[tid] = res;
            }
            __syncthreads();
            if (++k == a.max_inner) break;
            if (half() <= tin2 || s_bad) break;
            z = product(bt, nullptr, vb, false);
            const double beta = scalar(va, z, [&](double rzn) {
                const double v = rzn / rz;
                rz = rzn;
                return v;
            });
            if (!dots) d = z[tid] + (T)beta * d;
        }
    }
    if (rank == 0 && !dots) {
        a.y[tid] = y;
        if (tid == 0) ctl->inner_iters += k;
    }
    cl.sync();   // a CTA whose wait ran out stays until nobody sends to it (the others' waits end too)
}

// The kernel for a padded sketch size (its data fits the cluster's registers),
// null where there is none.
template <typename T>
const void* inner_kernel(int64_t sp) {
    switch (sp) {
        case 128: return (const void*)k_inner<T, 8>;
        case 256: return (const void*)k_inner<T, 16>;
        case 384:
            if constexpr (sizeof(T) == 4) return (const void*)k_inner<T, 24>;
            return nullptr;
        default: return nullptr;
    }
}

cudaLaunchConfig_t inner_config(msp_ctx* ctx, int64_t sp, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kInnerCtas);
    cfg.blockDim = dim3((unsigned)(sp + kDotThreads));
    cfg.stream = ctx->stream;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = kInnerCtas;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <typename T>
msp_status launch_inner(msp_ctx* ctx, InnerArgs<T>& a, int64_t sp) {
    const void* kern = inner_kernel<T>(sp);
    MSP_CUDA_TRY(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = inner_config(ctx, sp, &attr);
    void* args[] = {&a};
    ++ctx->launches;
    MSP_CUDA_TRY(ctx, cudaLaunchKernelExC(&cfg, kern, args));
    return MSP_OK;
}

// The level-2 step of an iteration: k_level2 whole (a direct level 2, no formed
// operator), or k_inner between its two parts.
template <typename T, typename TC>
msp_status launch_level2(msp_ctx* ctx, L2Args<T, TC>& a, int G, InnerArgs<T>& in) {
    if (!in.H || a.max_inner <= 0) return launch_level2(ctx, a, G);
    a.phase = PHASE_FRONT;
    msp_status st = launch_level2(ctx, a, G);
    if (st == MSP_OK) st = launch_inner<T>(ctx, in, a.s_pad);
    a.phase = PHASE_BACK;
    if (st == MSP_OK) st = launch_level2(ctx, a, G);
    a.phase = PHASE_ALL;
    return st;
}

struct Workspace {
    void* part;
    void* vecs;
    double* dpart;
    void* level1;   // x r q p p' z (n_pad each)
    double* gpart;  // A-pass partials
    float* qpart;   // packed A pass: nt x n_pad slot partials (or null)
    int64_t n_pad;
};

template <typename T>
msp_status get_workspace(msp_ctx* ctx, int64_t n, int64_t sp, int G, int Gg, bool packed,
                         Workspace* ws) {
    size_t ts = sizeof(T);
    const int64_t n_pad = round_up(n, 128);
    const int64_t nt = n_pad / 128;
    size_t b_part = round_up((int64_t)G * sp * ts, 256);
    size_t b_vecs = round_up(5 * sp * ts, 256);
    size_t b_dpart = round_up((int64_t)G * 4 * 8, 256);
    size_t b_l1 = round_up(6 * n_pad * ts, 256);
    size_t b_gp = round_up((int64_t)Gg * 8, 256);
    size_t b_qp = packed ? round_up(nt * n_pad * 4, 256) : 0;
    void* scr = nullptr;
    MSP_TRY(msp_scratch(ctx, b_part + b_vecs + b_dpart + b_l1 + b_gp + b_qp, &scr));
    char* c = (char*)scr;
    ws->part = c; c += b_part;
    ws->vecs = c; c += b_vecs;
    ws->dpart = (double*)c; c += b_dpart;
    ws->level1 = c; c += b_l1;
    ws->gpart = (double*)c; c += b_gp;
    ws->qpart = packed ? (float*)c : nullptr;
    ws->n_pad = n_pad;
    return MSP_OK;
}

template <typename T, typename TC>
void fill_l2(L2Args<T, TC>& a, const msp_factor_s* f, int64_t n, const Workspace& ws, CtlBlock* ctl) {
    const int64_t sp = f->s_pad;
    a.n = n;
    a.s_pad = sp;
    // BF16 preconditioner data: the factor's rounded copies of C and W
    a.C = (const TC*)(f->data == MSP_BF16 ? f->Cb : f->sk->C);
    a.W = (const TC*)(f->data == MSP_BF16 ? f->Wb : f->W);
    a.B = (const T*)f->B;
    a.Bt = (const T*)f->Bt;
    a.lam_t = (T)f->lam_tilde;
    a.ctl = ctl;
    a.part = (T*)ws.part;
    T* v = (T*)ws.vecs;
    a.gvec = v;
    a.uvec = v + sp;
    a.tvec = v + 2 * sp;
    a.zvec = v + 3 * sp;
    a.wdvec = v + 4 * sp;
    a.dpart = ws.dpart;
}

// after the options are in `a`
template <typename T, typename TC>
InnerArgs<T> fill_inner(const msp_factor_s* f, const L2Args<T, TC>& a) {
    InnerArgs<T> in;
    std::memset(&in, 0, sizeof in);
    if (!f->H || f->data == MSP_BF16) return in;
    in.H = (const T*)f->H;
    in.Hlo = sizeof(T) == 4 ? (const float*)f->H + f->s_pad * f->s_pad : nullptr;
    in.B = a.B;
    in.Bt = a.Bt;
    in.g = a.gvec;
    in.y = a.zvec;
    in.inner_tol2 = a.inner_tol2;
    in.max_inner = a.max_inner;
    in.ctl = a.ctl;
    return in;
}

// The level-2 grid: one block per SM (a thread per block partial in the
// column sums, so at most kThreads).
int level2_grid(msp_ctx* ctx) { return std::min(ctx->num_sms, kThreads); }
int gemv_grid(msp_ctx* ctx) { return ctx->num_sms * 8; }

// ------------------------------------------------ level-1 graph replay
//
// One level-1 iteration is two launches whose arguments do not change from
// one iteration to the next (the A pass and the cooperative level-2 kernel;
// the scalars travel through the control block). It is captured once into a
// CUDA graph and replayed, which removes the per-launch host work and most
// of the gap between the two kernels. The executable is cached in the
// context under a key of everything the launches were built from (argument
// structs, buffers, grid sizes); any change rebuilds it.

constexpr int kL1Timed = 2;     // event-record nodes of a timed iteration graph

// Captures iter(true) (launches on ctx->stream, redirected to the capture
// stream) as the context's level-1 graph for `key`. With `timed`, iter puts
// an event-record node before the A pass and one between the A pass and the
// level-2 kernel (ctx->events[0..1]), found again here by their events so
// that each replay can point them at fresh events. Leaves ctx->l1_exec null
// where capture is not possible; the caller then launches on the stream.
template <typename F>
msp_status ensure_l1_graph(msp_ctx* ctx, const void* key, size_t klen, bool timed, F&& iter) {
    if (ctx->l1_exec && ctx->l1_key_len == klen && std::memcmp(ctx->l1_key, key, klen) == 0)
        return MSP_OK;
    msp_l1_graph_release(ctx);
    if (klen > sizeof(ctx->l1_key)) return MSP_OK;
    if (!ctx->cap_stream &&
        cudaStreamCreateWithFlags(&ctx->cap_stream, cudaStreamNonBlocking) != cudaSuccess) {
        cudaGetLastError();
        ctx->cap_stream = nullptr;
        return MSP_OK;
    }
    if (cudaStreamBeginCapture(ctx->cap_stream, cudaStreamCaptureModeRelaxed) != cudaSuccess) {
        cudaGetLastError();
        return MSP_OK;
    }
    const cudaStream_t saved = ctx->stream;
    const int64_t l0 = ctx->launches;
    ctx->stream = ctx->cap_stream;
    const msp_status st = iter(true);
    ctx->stream = saved;
    cudaGraph_t graph = nullptr;
    const cudaError_t ce = cudaStreamEndCapture(ctx->cap_stream, &graph);
    const int kernels = (int)(ctx->launches - l0);
    ctx->launches = l0;
    bool ok = st == MSP_OK && ce == cudaSuccess && graph != nullptr;
    cudaGraphNode_t evn[kL1Timed] = {};
    if (ok && timed) {
        size_t nn = 0;
        ok = cudaGraphGetNodes(graph, nullptr, &nn) == cudaSuccess && nn > 0 && nn <= 64;
        cudaGraphNode_t nodes[64];
        if (ok) ok = cudaGraphGetNodes(graph, nodes, &nn) == cudaSuccess;
        for (size_t i = 0; ok && i < nn; ++i) {
            cudaGraphNodeType ty;
            if (cudaGraphNodeGetType(nodes[i], &ty) != cudaSuccess) { ok = false; break; }
            if (ty != cudaGraphNodeTypeEventRecord) continue;
            cudaEvent_t ev = nullptr;
            if (cudaGraphEventRecordNodeGetEvent(nodes[i], &ev) != cudaSuccess) { ok = false; break; }
            for (int k = 0; k < kL1Timed; ++k)
                if (ev == ctx->events[k]) evn[k] = nodes[i];
        }
        for (int k = 0; ok && k < kL1Timed; ++k) ok = evn[k] != nullptr;
    }
    if (ok && cudaGraphInstantiate(&ctx->l1_exec, graph, 0) != cudaSuccess) {
        ctx->l1_exec = nullptr;
        ok = false;
    }
    if (!ok) {
        if (graph) cudaGraphDestroy(graph);
        cudaGetLastError();
        return MSP_OK;
    }
    ctx->l1_graph = graph;
    std::memcpy(ctx->l1_key, key, klen);
    ctx->l1_key_len = klen;
    for (int k = 0; k < kL1Timed; ++k) ctx->l1_ev_nodes[k] = evn[k];
    ctx->l1_kernels = kernels;
    return MSP_OK;
}

// Replays one level-1 iteration. Timed: the graph's two event-record nodes
// get fresh events b (before the A pass) and e (after it); the A pass is
// the entry (b, e), and the level-2 kernel of the iteration before, whose
// end the new b marks, the entry (e_prev, b): two events per iteration.
// *l2_open holds e of the last replay until then (-1: none); the spare
// events past the pool stand in once it is used up. Already queued replays
// keep their events.
msp_status replay_l1(msp_ctx* ctx, Profiler& pr, int* l2_open) {
    if (pr.on) {
        cudaEvent_t eb = ctx->events[ctx->n_events - 2], ee = ctx->events[ctx->n_events - 1];
        int ib = -1, ie = -1;
        const bool fresh = pr.take(&eb, &ib) && pr.take(&ee, &ie);
        if (!fresh) {
            eb = ctx->events[ctx->n_events - 2];
            ee = ctx->events[ctx->n_events - 1];
        }
        MSP_CUDA_TRY(ctx, cudaGraphExecEventRecordNodeSetEvent(ctx->l1_exec, ctx->l1_ev_nodes[0], eb));
        MSP_CUDA_TRY(ctx, cudaGraphExecEventRecordNodeSetEvent(ctx->l1_exec, ctx->l1_ev_nodes[1], ee));
        if (fresh) {
            if (*l2_open >= 0) pr.add(1, *l2_open, ib);
            pr.add(0, ib, ie);
        }
        *l2_open = fresh ? ie : -1;
    }
    MSP_CUDA_TRY(ctx, cudaGraphLaunch(ctx->l1_exec, ctx->stream));
    ctx->launches += ctx->l1_kernels;
    ++ctx->l1_graph_iters;
    return MSP_OK;
}

// Ends the timing chain after the last replay of a check interval: an event
// on the stream closes the open level-2 entry.
msp_status close_l1_chain(msp_ctx* ctx, Profiler& pr, int* l2_open) {
    if (!pr.on || *l2_open < 0) return MSP_OK;
    cudaEvent_t ev;
    int idx;
    if (pr.take(&ev, &idx)) {
        MSP_CUDA_TRY(ctx, cudaEventRecord(ev, ctx->stream));
        pr.add(1, *l2_open, idx);
    }
    *l2_open = -1;
    return MSP_OK;
}

template <typename T, typename TC = T>
msp_status krylov_solve_t(msp_ctx* ctx, const msp_factor_s* f, const void* A, msp_dtype dt,
                          int64_t n, int64_t lda, double lambda, const T* rhs, T* sol,
                          double tol_rel, int max_outer, const msp_opts* o, int* iters,
                          int* inner_iters, ProfSlot* prof, const float* packed) {
    const int G = level2_grid(ctx), Gg = gemv_grid(ctx);
    const bool use_packed = (packed != nullptr) && (sizeof(T) == 4);
    Profiler pr;
    pr.ctx = ctx;
    pr.on = (prof != nullptr) && o->profile;
    if (pr.on) MSP_TRY(msp_profiler_reserve(ctx, 4096));
    Workspace ws;
    MSP_TRY(get_workspace<T>(ctx, n, f->s_pad, G, Gg, use_packed, &ws));
    const int64_t np = ws.n_pad;
    T* x = (T*)ws.level1;
    T* r = x + np;
    T* q = r + np;
    T* p = q + np;
    T* z = p + 2 * np;      // p: two buffers (the packed A pass writes them in turn)
    CtlBlock* ctl = (CtlBlock*)ctx->ctl;
    MSP_CUDA_TRY(ctx, cudaMemsetAsync(ctl, 0, sizeof(CtlBlock), ctx->stream));
    // all the level-1 vectors, pads included (p and z must be zero past n)
    MSP_CUDA_TRY(ctx, cudaMemsetAsync(x, 0, 6 * np * sizeof(T), ctx->stream));
    MSP_CUDA_TRY(ctx, cudaMemcpyAsync(r, rhs, n * sizeof(T), cudaMemcpyDeviceToDevice, ctx->stream));

    // zeroed bytes (padding included): the struct is part of the graph key
    L2Args<T, TC> a;
    std::memset(&a, 0, sizeof a);
    fill_l2(a, f, n, ws, ctl);
    a.tol_rel2 = tol_rel * tol_rel;
    a.inner_tol2 = o->inner_tol * o->inner_tol;
    a.max_inner = o->max_inner;
    a.x = x; a.r = r; a.q = q; a.p = p; a.z = z;
    a.qpart = use_packed ? ws.qpart : nullptr;
    a.q_slots = (int)(np / 128);
    a.q_ld = np;
    a.p_ld = np;
    a.dq = use_packed ? ws.gpart : nullptr;
    a.n_dq = ctx->num_sms;
    a.lam = (T)lambda;
    a.prog = (volatile int*)((char*)ctx->host_flags + 192);
    a.prog[0] = 0;
    a.prog[1] = 0;
    a.mode = MODE_INIT;
    InnerArgs<T> in = fill_inner(f, a);
    MSP_TRY(launch_level2(ctx, a, G, in));
    a.mode = MODE_ITER;

    const bool vec = (lda % (16 / dtype_size(dt)) == 0) &&
                     ((uintptr_t)A % 16 == 0) && (n % (16 / dtype_size(dt)) == 0);
    // one level-1 iteration: the A pass q = (A + lam I) p, then the level-2
    // kernel (the step, SolveM1, the new direction); `cap`: inside a graph
    // capture, where event-record nodes take the profiler's place
    auto mark = [&](bool cap, int k) -> msp_status {
        if (!pr.on) return MSP_OK;
        if (cap) {
            // event-record nodes before the A pass and between the launches
            if (k < kL1Timed)
                MSP_CUDA_TRY(ctx, cudaEventRecordWithFlags(ctx->events[k], ctx->stream, cudaEventRecordExternal));
            return MSP_OK;
        }
        return (k & 1) ? pr.end() : pr.begin(k >> 1);
    };
    auto iteration = [&](bool cap) -> msp_status {
        MSP_TRY(mark(cap, 0));
        if (use_packed) {
            MSP_TRY(msp_symv_packed(ctx, packed, n, (float)lambda, (const float*)z, (float*)p, ws.dpart, G, ws.qpart,
                                    ws.gpart, ctx->num_sms));
        } else {
            if (dt == MSP_F32) {
                if (vec) k_gemv<float, T, true><<<Gg, 256, 0, ctx->stream>>>((const float*)A, lda, n, lambda, p, q, ws.gpart, ctl);
                else k_gemv<float, T, false><<<Gg, 256, 0, ctx->stream>>>((const float*)A, lda, n, lambda, p, q, ws.gpart, ctl);
            } else {
                if (vec) k_gemv<double, T, true><<<Gg, 256, 0, ctx->stream>>>((const double*)A, lda, n, lambda, p, q, ws.gpart, ctl);
                else k_gemv<double, T, false><<<Gg, 256, 0, ctx->stream>>>((const double*)A, lda, n, lambda, p, q, ws.gpart, ctl);
            }
            MSP_CHECK_LAUNCH(ctx);
        }
        MSP_TRY(mark(cap, 1));
        MSP_TRY(mark(cap, 2));
        MSP_TRY(launch_level2(ctx, a, G, in));
        MSP_TRY(mark(cap, 3));
        return MSP_OK;
    };
    bool graphed = false;
    if (ctx->l1_graphs) {
        struct Key {
            int tag, dt, use_packed, vec, G, Gg, timed, pad;
            const void* A;
            int64_t lda;
            const float* packed;
            double lambda;
            const void* qpart;
            const void* gpart;
            const void* H;
            L2Args<T, TC> a;
        } key;
        static_assert(sizeof(Key) <= sizeof(ctx->l1_key), "level-1 graph key too large");
        std::memset(&key, 0, sizeof key);
        key.tag = (int)(10 * sizeof(T) + sizeof(TC));
        key.dt = (int)dt;
        key.use_packed = use_packed;
        key.vec = vec;
        key.G = G;
        key.Gg = Gg;
        key.timed = pr.on;
        key.A = A;
        key.lda = lda;
        key.packed = packed;
        key.lambda = lambda;
        key.qpart = ws.qpart;
        key.gpart = ws.gpart;
        key.H = in.H;
        std::memcpy(&key.a, &a, sizeof a);
        MSP_TRY(ensure_l1_graph(ctx, &key, sizeof key, pr.on, iteration));
        graphed = ctx->l1_exec != nullptr;
    }
    int* hf = (int*)ctx->host_flags;
    const int check = std::max(1, o->check_every);
    // the packed A pass finds an indefinite or non-finite r^T w of the iteration
    // before it: after the last allowed iteration one more pass looks at that one's
    auto last_look = [&]() -> msp_status {
        if (!use_packed) return MSP_OK;
        return msp_symv_packed(ctx, packed, n, (float)lambda, (const float*)z, (float*)p, ws.dpart, G, ws.qpart,
                               ws.gpart, ctx->num_sms);
    };
    // profiler entries of iterations known to have run to completion with
    // work (every iteration before a check that found no flag): read while
    // the next interval runs, not after it
    int settled = 0, l2_open = -1;
    // a program that asked for blocking or yielding synchronisation wants the core for
    // itself: there the host sleeps in a stream synchronisation per check interval
    unsigned int flags = 0;
    const bool spin = cudaGetDeviceFlags(&flags) != cudaSuccess ||
                      !(flags & (cudaDeviceScheduleBlockingSync | cudaDeviceScheduleYield));
    if (!pr.on && spin) {
        // the device reports each iteration in pinned host words; the host keeps
        // at most `ahead` iterations queued and polls, so the stream never runs
        // dry between checks (a stream synchronisation every 8 iterations left it
        // idle for about 30 us) and few launches follow the converged one. The
        // poll ends when the stream has nothing left to do, whatever was reported.
        const int ahead = std::min(check, 4);
        int it = 0;
        while (it < max_outer && !a.prog[1]) {
            const int done = a.prog[0];
            if (it < done + ahead) {
                if (graphed) MSP_TRY(replay_l1(ctx, pr, &l2_open));
                else MSP_TRY(iteration(false));
                ++it;
                continue;
            }
            for (int spin = 0; a.prog[0] == done && !a.prog[1]; ++spin) {
                if ((spin & 1023) != 1023) continue;
                const cudaError_t e = cudaStreamQuery(ctx->stream);
                if (e == cudaSuccess) break;
                if (e != cudaErrorNotReady) MSP_CUDA_TRY(ctx, e);
            }
            // idle without a report: the launches ended early (an error word)
            if (a.prog[0] == done && !a.prog[1]) break;
        }
        if (it >= max_outer && !a.prog[1]) MSP_TRY(last_look());
    } else {
        for (int it = 0; it < max_outer;) {
            const int nrun = std::min(check, max_outer - it);
            for (int i = 0; i < nrun; ++i) {
                if (graphed) MSP_TRY(replay_l1(ctx, pr, &l2_open));
                else MSP_TRY(iteration(false));
            }
            if (graphed) MSP_TRY(close_l1_chain(ctx, pr, &l2_open));
            it += nrun;
            MSP_CUDA_TRY(ctx, cudaMemcpyAsync(hf, &ctl->done, 5 * sizeof(int), cudaMemcpyDeviceToHost,
                                              ctx->stream));
            MSP_TRY(pr.harvest(prof, 2, settled));
            MSP_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
            if (hf[0] || hf[1]) break;
            settled = pr.used;
            if (it >= max_outer) MSP_TRY(last_look());
        }
    }
    MSP_CUDA_TRY(ctx, cudaMemcpyAsync(hf, &ctl->done, 5 * sizeof(int), cudaMemcpyDeviceToHost,
                                      ctx->stream));
    MSP_CUDA_TRY(ctx, cudaMemcpyAsync(sol, x, n * sizeof(T), cudaMemcpyDeviceToDevice, ctx->stream));
    MSP_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    // the iterations that did work: ctl->iters counts them, and every launch
    // queued after the flag returned at once
    if (pr.on) MSP_TRY(pr.finish(prof, 2, 2 * hf[2]));
    // hf: done, error, iters, inner_iters, pad
    if (iters) *iters = hf[2];
    if (inner_iters) *inner_iters = hf[3];
    if (hf[1]) {
        const int e = hf[1];
        return msp_set_error(ctx, (msp_status)e, "level-1 iteration stopped with device status %d%s",
                             e, e == MSP_ETIMEOUT ? " (grid barrier timed out)" : "");
    }
    if (!hf[0]) return msp_set_error(ctx, MSP_ENOCONV, "no convergence in %d level-1 iterations",
                                     hf[2]);
    return MSP_OK;
}

}  // namespace

void msp_l1_graph_release(msp_ctx* ctx) {
    if (ctx->l1_exec) cudaGraphExecDestroy(ctx->l1_exec);
    if (ctx->l1_graph) cudaGraphDestroy(ctx->l1_graph);
    ctx->l1_exec = nullptr;
    ctx->l1_graph = nullptr;
    ctx->l1_key_len = 0;
    for (cudaGraphNode_t& nd : ctx->l1_ev_nodes) nd = nullptr;
    ctx->l1_kernels = 0;
}

extern "C" msp_status msp_set_level1_graphs(msp_ctx* ctx, int on) {
    if (!ctx) return msp_set_error(nullptr, MSP_EINVAL, "ctx is NULL");
    ctx->l1_graphs = on != 0;
    if (!ctx->l1_graphs) msp_l1_graph_release(ctx);
    return MSP_OK;
}

// The grid-barrier limit of this unit's kernels (the level-1 and level-2
// iterations) on the current device; 0 restores the default.
msp_status msp_grid_wait_limit_krylov(msp_ctx* ctx, unsigned long long ns) {
    const unsigned long long v = ns ? ns : msp::kWaitLimitNs;
    MSP_CUDA_TRY(ctx, cudaMemcpyToSymbol(msp::g_grid_wait_limit_ns, &v, sizeof v));
    return MSP_OK;
}

// Whether the level-2 iteration of a factor of this size runs on a formed
// operator (k_inner): a kernel for the size, and room for its cluster.
bool msp_inner_ok(msp_ctx* ctx, msp_dtype dt, int64_t sp) {
    const void* kern = dt == MSP_F32 ? inner_kernel<float>(sp) : inner_kernel<double>(sp);
    if (!kern) return false;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = inner_config(ctx, sp, &attr);
    int clusters = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters >= 1;
}

msp_status msp_krylov_solve(msp_ctx* ctx, const msp_factor_s* f, const void* A, msp_dtype dt,
                            int64_t n, int64_t lda, double lambda, const void* rhs, void* sol,
                            double tol_rel, int max_outer, const msp_opts* o, int* iters,
                            int* inner_iters, ProfSlot* prof, const float* packed) {
    if (f->dtype == MSP_F32 && f->data == MSP_BF16)
        return krylov_solve_t<float, __nv_bfloat16>(ctx, f, A, dt, n, lda, lambda, (const float*)rhs, (float*)sol,
                                                    tol_rel, max_outer, o, iters, inner_iters, prof, packed);
    if (f->dtype == MSP_F32)
        return krylov_solve_t<float>(ctx, f, A, dt, n, lda, lambda, (const float*)rhs, (float*)sol,
                                     tol_rel, max_outer, o, iters, inner_iters, prof, packed);
    return krylov_solve_t<double>(ctx, f, A, dt, n, lda, lambda, (const double*)rhs, (double*)sol,
                                  tol_rel, max_outer, o, iters, inner_iters, prof, nullptr);
}

// ---------------------------------------------------------------- profiler

// `pairs` event pairs plus four spare events at the end (the sinks of a
// timed level-1 graph once the pairs are used up)
msp_status msp_profiler_reserve(msp_ctx* ctx, int pairs) {
    const int want = 2 * pairs + 4;
    if (ctx->n_events >= want) return MSP_OK;
    for (int i = 0; i < ctx->n_events; ++i) cudaEventDestroy(ctx->events[i]);
    delete[] ctx->events;
    ctx->events = new cudaEvent_t[want];
    ctx->n_events = 0;
    for (int i = 0; i < want; ++i) {
        MSP_CUDA_TRY(ctx, cudaEventCreate(&ctx->events[i]));
        ctx->n_events = i + 1;
    }
    return MSP_OK;
}

msp_status Profiler::begin(int slot) {
    open = false;
    if (!on || used >= 4096 || next_ev + 2 > ctx->n_events - 4) return MSP_OK;
    slot_of[used] = slot;
    ev_b[used] = next_ev++;
    open = true;
    MSP_CUDA_TRY(ctx, cudaEventRecord(ctx->events[ev_b[used]], ctx->stream));
    return MSP_OK;
}

msp_status Profiler::end() {
    // closes the entry of the last begin() that went through
    if (!open) return MSP_OK;
    open = false;
    ev_e[used] = next_ev++;
    MSP_CUDA_TRY(ctx, cudaEventRecord(ctx->events[ev_e[used]], ctx->stream));
    ++used;
    return MSP_OK;
}

bool Profiler::take(cudaEvent_t* ev, int* idx) {
    if (!on || next_ev + 1 > ctx->n_events - 4) return false;
    *idx = next_ev++;
    *ev = ctx->events[*idx];
    return true;
}

void Profiler::add(int slot, int b, int e) {
    if (!on || used >= 4096) return;
    slot_of[used] = slot;
    ev_b[used] = b;
    ev_e[used] = e;
    ++used;
}

msp_status Profiler::harvest(ProfSlot* slots, int nslots, int upto) {
    if (!on) return MSP_OK;
    for (int i = harvested; i < upto && i < used; ++i) {
        float ms = 0.f;
        MSP_CUDA_TRY(ctx, cudaEventElapsedTime(&ms, ctx->events[ev_b[i]], ctx->events[ev_e[i]]));
        if (slot_of[i] < nslots) {
            slots[slot_of[i]].ms += ms;
            slots[slot_of[i]].launches += 1;
        }
        harvested = i + 1;
    }
    return MSP_OK;
}

msp_status Profiler::finish(ProfSlot* slots, int nslots, int keep) {
    if (!on) return MSP_OK;
    MSP_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    MSP_TRY(harvest(slots, nslots, (keep >= 0 && keep < used) ? keep : used));
    used = 0;
    harvested = 0;
    next_ev = 0;
    return MSP_OK;
}

msp_status msp_solve_m1_impl(msp_ctx* ctx, const msp_factor_s* f, const void* r, void* w,
                             const msp_opts* o, int* inner_iters) {
    const int64_t n = f->sk->n;
    const int G = level2_grid(ctx), Gg = gemv_grid(ctx);
    CtlBlock* ctl = (CtlBlock*)ctx->ctl;
    MSP_CUDA_TRY(ctx, cudaMemsetAsync(ctl, 0, sizeof(CtlBlock), ctx->stream));
    int* hf = (int*)ctx->host_flags;
    if (f->dtype == MSP_F32 && f->data == MSP_BF16) {
        Workspace ws;
        MSP_TRY(get_workspace<float>(ctx, n, f->s_pad, G, Gg, false, &ws));
        L2Args<float, __nv_bfloat16> a{};
        fill_l2(a, f, n, ws, ctl);
        a.inner_tol2 = o->inner_tol * o->inner_tol;
        a.max_inner = o->max_inner;
        a.r = (float*)r;
        a.z = (float*)w;
        a.mode = MODE_APPLY;
        auto in = fill_inner(f, a);
        MSP_TRY(launch_level2(ctx, a, G, in));
    } else if (f->dtype == MSP_F32) {
        Workspace ws;
        MSP_TRY(get_workspace<float>(ctx, n, f->s_pad, G, Gg, false, &ws));
        L2Args<float> a{};
        fill_l2(a, f, n, ws, ctl);
        a.inner_tol2 = o->inner_tol * o->inner_tol;
        a.max_inner = o->max_inner;
        a.r = (float*)r;
        a.z = (float*)w;
        a.mode = MODE_APPLY;
        auto in = fill_inner(f, a);
        MSP_TRY(launch_level2(ctx, a, G, in));
    } else {
        Workspace ws;
        MSP_TRY(get_workspace<double>(ctx, n, f->s_pad, G, Gg, false, &ws));
        L2Args<double> a{};
        fill_l2(a, f, n, ws, ctl);
        a.inner_tol2 = o->inner_tol * o->inner_tol;
        a.max_inner = o->max_inner;
        a.r = (double*)r;
        a.z = (double*)w;
        a.mode = MODE_APPLY;
        auto in = fill_inner(f, a);
        MSP_TRY(launch_level2(ctx, a, G, in));
    }
    MSP_CUDA_TRY(ctx, cudaMemcpyAsync(hf, &ctl->done, 5 * sizeof(int), cudaMemcpyDeviceToHost,
                                      ctx->stream));
    MSP_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    if (inner_iters) *inner_iters = hf[3];
    if (hf[1]) return msp_set_error(ctx, (msp_status)hf[1], "SolveM1: device status %d", hf[1]);
    return MSP_OK;
}

namespace {

// Error-free transformations (Knuth's TwoSum; the FMA form of Dekker's
// TwoProduct): a + b = s + e and a b = p + e exactly in FP64.
__device__ inline void two_sum(double a, double b, double& s, double& e) {
    s = a + b;
    const double bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
__device__ inline void two_prod(double a, double b, double& p, double& e) {
    p = a * b;
    e = fma(a, b, -p);
}
// (hi, lo) += (p, q), a double-double sum (hi, lo) renormalised
__device__ inline void dd_add(double& hi, double& lo, double p, double q) {
    double s, e;
    two_sum(hi, p, s, e);
    e += lo + q;
    hi = s + e;
    lo = e - (hi - s);
}

// x = xh + xl with xh = fl32(x), xl = fl32(x - xh) (x - xh exact in FP64):
// |x - xh - xl| <= 2^-48 |x|.
__global__ void k_split_x(const double* __restrict__ x, int64_t n, float* __restrict__ xh, float* __restrict__ xl) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const double v = x[j];
        const float h = (float)v;
        xh[j] = h;
        xl[j] = (float)(v - (double)h);
    }
}

// (hi, lo) += p + t (|t| small): TwoSum (Knuth) of hi and p, the error, lo
// and t added, then renormalised by Fast2Sum (Dekker) so that |lo| stays
// within half an ulp of hi; each call adds at most about 2^-47 |hi| of error.
__device__ __forceinline__ void ff_acc(float& hi, float& lo, float p, float t) {
    const float s = __fadd_rn(hi, p);
    const float bp = __fsub_rn(s, hi);
    float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(p, bp));
    e = __fadd_rn(e, __fadd_rn(lo, t));
    hi = __fadd_rn(s, e);
    lo = __fsub_rn(e, __fsub_rn(hi, s));
}

// out = b - (A + lam I) x for an FP32 A in float-float arithmetic on the FP32
// pipe (the FP64 pipe of this part, two FMAs per clock per SM, held the FP64
// version to a third of the HBM rate). Per element: a xh exactly as p + e
// (TwoProd by FMA), a xl + e rounded (at most about 2^-47 |a x|), both added
// to a per-lane float-float pair (ff_acc). Four pairs per lane (one per
// float4 component), n / 128 elements each; the pairs are added in FP64 in a
// fixed order. Error at most about (n / 128 + 2) 2^-47 sum_j |a_ij x_j|
// (2^-40 at n = 16384), with the split of x: far below the backward errors
// the refinement resolves (1e-10 ~ 2^-33). |out|^2 into *norm2 as k_matvec64.
// Requires lda, n multiples of 4 and 16-byte aligned A. SPLIT: x is split by each
// block into shared memory (n <= kSplitMax) and xh, xl are not read: one launch for a
// small system, where the launches and blocks are the time (20.5 us a call at n = 1000
// with k_split_x and 1216 blocks, 8 to 10 us with this and a block per 8 rows); each block then
// pays four FP64-pipe conversions per 32 entries, which the split kernel's 2 us outweigh
// from about 1600 entries on. us a call without and with this: 13 to 14 and 10.0 at n = 1100, 13.1
// and 12.3 at 1300, 14.3 and 13.7 at 1500, 15.1 and 15.1 at 1700, 15.9 and 17.7 at 2000.
constexpr int kSplitMax = 1536;

template <bool SPLIT>
__global__ void __launch_bounds__(256, 2) k_matvec64_ff(const float* __restrict__ A, int64_t lda, int64_t n,
                                                    double lam, const float* __restrict__ xh,
                                                    const float* __restrict__ xl, const double* __restrict__ x,
                                                    const double* __restrict__ b, double* __restrict__ out,
                                                    double* __restrict__ part, unsigned int* counter,
                                                    double* norm2) {
    __shared__ double red[32];
    __shared__ bool am_last;
    __shared__ __align__(16) float sx[2][SPLIT ? kSplitMax : 4];
    if constexpr (SPLIT) {
        for (int j = threadIdx.x; j < (int)n; j += 256) {
            const double v = x[j];
            const float h = (float)v;
            sx[0][j] = h;
            sx[1][j] = (float)(v - (double)h);
        }
        __syncthreads();
        xh = sx[0];
        xl = sx[1];
    }
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    double nn = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += warps) {
        const float* row = A + i * lda;
        float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
        int64_t j = (int64_t)lane * 4;
        for (; j + 128 < n; j += 256) {
            const float4 a0 = __ldcs(reinterpret_cast<const float4*>(row + j));
            const float4 a1 = __ldcs(reinterpret_cast<const float4*>(row + j + 128));
            const float4 h0 = (*reinterpret_cast<const float4*>(xh + j));
            const float4 h1 = (*reinterpret_cast<const float4*>(xh + j + 128));
            const float4 l0 = (*reinterpret_cast<const float4*>(xl + j));
            const float4 l1 = (*reinterpret_cast<const float4*>(xl + j + 128));
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float hv[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
            const float lv[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float p = __fmul_rn(av[k], hv[k]);
                const float e = __fmaf_rn(av[k], hv[k], -p);
                ff_acc(hi[k & 3], lo[k & 3], p, __fmaf_rn(av[k], lv[k], e));
            }
        }
        for (; j < n; j += 128) {
            const float4 a0 = __ldcs(reinterpret_cast<const float4*>(row + j));
            const float4 h0 = (*reinterpret_cast<const float4*>(xh + j));
            const float4 l0 = (*reinterpret_cast<const float4*>(xl + j));
            const float av[4] = {a0.x, a0.y, a0.z, a0.w};
            const float hv[4] = {h0.x, h0.y, h0.z, h0.w};
            const float lv[4] = {l0.x, l0.y, l0.z, l0.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float p = __fmul_rn(av[k], hv[k]);
                const float e = __fmaf_rn(av[k], hv[k], -p);
                ff_acc(hi[k], lo[k], p, __fmaf_rn(av[k], lv[k], e));
            }
        }
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) acc += (double)hi[k] + (double)lo[k];
        acc = msp::warp_sum(acc);
        if (lane == 0) {
            double v = acc + lam * x[i];
            if (b) v = b[i] - v;
            out[i] = v;
            nn += v * v;
        }
    }
    if (!norm2) return;
    double tot = block_sum(nn, red);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = tot;
        __threadfence();
        unsigned int t = atomicAdd(counter, 1u);
        am_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    double all = sum_parts(part, 1, gridDim.x, red);
    if (threadIdx.x == 0) {
        *counter = 0;
        *norm2 = all;
    }
}

// out = b - (A + lam I) x with double-double accumulation: every product
// and sum error-free transformed, rounded to FP64 once per row. Its error is
// a few u |r_i| + u^2 sum_j |A_ij x_j| instead of u sum_j |A_ij x_j|, so the
// residual of an ill-conditioned system stays resolved below the FP64
// accumulation floor. |out|^2 into *norm2 as k_matvec64.
template <typename TA>
__global__ void __launch_bounds__(256) k_matvec64_dd(const TA* __restrict__ A, int64_t lda, int64_t n, double lam,
                                                    const double* __restrict__ x, const double* __restrict__ b,
                                                    double* __restrict__ out, double* __restrict__ part,
                                                    unsigned int* counter, double* norm2) {
    __shared__ double red[32];
    __shared__ bool am_last;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    double nn = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += warps) {
        const TA* row = A + i * lda;
        double hi = 0.0, lo = 0.0;
        for (int64_t j = lane; j < n; j += 32) {
            double p, e;
            two_prod(wide64(__ldcs(&row[j])), x[j], p, e);
            dd_add(hi, lo, p, e);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ph = __shfl_xor_sync(0xffffffffu, hi, o);
            const double pl = __shfl_xor_sync(0xffffffffu, lo, o);
            dd_add(hi, lo, ph, pl);
        }
        if (lane == 0) {
            double p, e;
            two_prod(lam, x[i], p, e);
            dd_add(hi, lo, p, e);
            double v = hi + lo;
            if (b) {
                double rh = b[i], rl = 0.0;
                dd_add(rh, rl, -hi, -lo);
                v = rh + rl;
            }
            out[i] = v;
            nn += v * v;
        }
    }
    double tot = block_sum(nn, red);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = tot;
        __threadfence();
        unsigned int t = atomicAdd(counter, 1u);
        am_last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    double all = sum_parts(part, 1, gridDim.x, red);
    if (threadIdx.x == 0) {
        *counter = 0;
        if (norm2) *norm2 = all;
    }
}

}  // namespace

msp_status msp_matvec64(msp_ctx* ctx, const void* A, msp_dtype dt, int64_t n, int64_t lda,
                        double lambda, const double* x, const double* b, double* out,
                        double* norm2_out_dev, bool compensated) {
    const int Gg = gemv_grid(ctx);
    void* scr = nullptr;
    const size_t b_part = round_up((int64_t)Gg * 8, 256), b_x = round_up(n * 4, 256);
    MSP_TRY(msp_scratch(ctx, b_part + 2 * b_x + 256, &scr));
    CtlBlock* ctl = (CtlBlock*)ctx->ctl;
    if (dt == MSP_BF16) {
        // BF16 A (the matvec of a BF16-stored matrix, e.g. to measure its
        // rounding against an FP32 or FP64 copy)
        if (compensated)
            k_matvec64_dd<__nv_bfloat16><<<Gg, 256, 0, ctx->stream>>>((const __nv_bfloat16*)A, lda, n, lambda, x, b,
                                                                      out, (double*)scr, &ctl->last_block_counter,
                                                                      norm2_out_dev);
        else
            k_matvec64<__nv_bfloat16, false><<<Gg, 256, 0, ctx->stream>>>((const __nv_bfloat16*)A, lda, n, lambda, x,
                                                                          b, out, (double*)scr,
                                                                          &ctl->last_block_counter, norm2_out_dev);
        MSP_CHECK_LAUNCH(ctx);
        return MSP_OK;
    }
    if (compensated) {
        if (dt == MSP_F32)
            k_matvec64_dd<float><<<Gg, 256, 0, ctx->stream>>>((const float*)A, lda, n, lambda, x, b, out,
                                                              (double*)scr, &ctl->last_block_counter,
                                                              norm2_out_dev);
        else
            k_matvec64_dd<double><<<Gg, 256, 0, ctx->stream>>>((const double*)A, lda, n, lambda, x, b, out,
                                                               (double*)scr, &ctl->last_block_counter,
                                                               norm2_out_dev);
        MSP_CHECK_LAUNCH(ctx);
        return MSP_OK;
    }
    const bool vec = (dt == MSP_F32) && (lda % 4 == 0) && (n % 4 == 0) &&
                     ((uintptr_t)A % 16 == 0) && ((uintptr_t)x % 16 == 0);
    if (dt == MSP_F32) {
        if (vec) {
            // a row per warp: no more blocks than rows / 8
            const int grid = (int)std::min<int64_t>(Gg, (n + 7) / 8);
            // with x split by every block no block may write into x meanwhile (y over x, as
            // the split kernel ahead of the product allows)
            const uintptr_t xa = (uintptr_t)x, oa = (uintptr_t)out;
            const bool apart = xa + (uintptr_t)n * 8 <= oa || oa + (uintptr_t)n * 8 <= xa;
            if (n <= kSplitMax && apart) {
                k_matvec64_ff<true><<<grid, 256, 0, ctx->stream>>>((const float*)A, lda, n, lambda, nullptr, nullptr, x, b,
                                                                   out, (double*)scr, &ctl->last_block_counter,
                                                                   norm2_out_dev);
                MSP_CHECK_LAUNCH(ctx);
                return MSP_OK;
            }
            float* xh = (float*)((char*)scr + b_part);
            float* xl = (float*)((char*)scr + b_part + b_x);
            k_split_x<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4 * ctx->num_sms), 256, 0, ctx->stream>>>(
                x, n, xh, xl);
            MSP_CHECK_LAUNCH(ctx);
            k_matvec64_ff<false><<<grid, 256, 0, ctx->stream>>>((const float*)A, lda, n, lambda, xh, xl, x, b, out,
                                                                (double*)scr, &ctl->last_block_counter,
                                                                norm2_out_dev);
        } else
            k_matvec64<float, false><<<Gg, 256, 0, ctx->stream>>>((const float*)A, lda, n, lambda, x, b,
                                                                  out, (double*)scr,
                                                                  &ctl->last_block_counter, norm2_out_dev);
    } else {
        k_matvec64<double, false><<<Gg, 256, 0, ctx->stream>>>((const double*)A, lda, n, lambda, x, b,
                                                               out, (double*)scr,
                                                               &ctl->last_block_counter, norm2_out_dev);
    }
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}
// ------------------------------------------------------------ vector ops

namespace {

// |v|^2 of an FP64 vector, one block, fixed order.
__global__ void k_norm2(const double* __restrict__ v, int64_t n, double* __restrict__ out) {
    __shared__ double red[32];
    double acc = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) acc += v[i] * v[i];
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) *out = acc;
}

__global__ void k_dot(const double* __restrict__ x, const double* __restrict__ y, int64_t n, double scale,
                      double* __restrict__ out) {
    __shared__ double red[32];
    double acc = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) acc += x[i] * y[i];
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) *out = scale * acc;
}

// dst = (T)(src / sqrt(*nrm2)) (0 if the norm is 0)
template <typename T>
__global__ void k_scale_cast(const double* __restrict__ src, const double* __restrict__ nrm2,
                             int64_t n, T* __restrict__ dst) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = *nrm2 > 0.0 ? 1.0 / sqrt(*nrm2) : 0.0;
    dst[i] = (T)(src[i] * s);
}

// x (+)= sqrt(*nrm2) * (double)d
template <typename T>
__global__ void k_axpy_back(double* __restrict__ x, const T* __restrict__ d,
                            const double* __restrict__ nrm2, int64_t n, int accumulate) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double v = sqrt(*nrm2) * (double)d[i];
    x[i] = accumulate ? x[i] + v : v;
}

}  // namespace

msp_status msp_norm2(msp_ctx* ctx, const double* v, int64_t n, double* out_dev) {
    k_norm2<<<1, 1024, 0, ctx->stream>>>(v, n, out_dev);
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

extern "C" msp_status msp_dot(msp_ctx* ctx, const double* x, const double* y, int64_t n, double scale,
                              double* out) {
    if (!ctx) return msp_set_error(nullptr, MSP_EINVAL, "ctx is NULL");
    if (!x || !y || !out || n < 1) return msp_set_error(ctx, MSP_EINVAL, "dot: bad argument");
    msp::DeviceGuard g(ctx->device);
    k_dot<<<1, 1024, 0, ctx->stream>>>(x, y, n, scale, out);
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

msp_status msp_scale_cast(msp_ctx* ctx, const double* src, const double* nrm2, int64_t n,
                          msp_dtype dt, void* dst) {
    unsigned g = (unsigned)((n + 255) / 256);
    if (dt == MSP_F32) k_scale_cast<float><<<g, 256, 0, ctx->stream>>>(src, nrm2, n, (float*)dst);
    else k_scale_cast<double><<<g, 256, 0, ctx->stream>>>(src, nrm2, n, (double*)dst);
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

msp_status msp_axpy_back(msp_ctx* ctx, double* x, const void* d, msp_dtype dt, const double* nrm2,
                         int64_t n, int accumulate) {
    unsigned g = (unsigned)((n + 255) / 256);
    if (dt == MSP_F32) k_axpy_back<float><<<g, 256, 0, ctx->stream>>>(x, (const float*)d, nrm2, n, accumulate);
    else k_axpy_back<double><<<g, 256, 0, ctx->stream>>>(x, (const double*)d, nrm2, n, accumulate);
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}
