// RBF kernel matrices and the adjoint of their length scale, on sm_103a.
//
// Coordinates are carried as exact FP32 pairs p = hi + lo, so a coordinate
// difference (hi_i - hi_j) + (lo_i - lo_j) is accurate to a few FP32 ulps of
// the difference itself (not of the coordinates): d_ij^2 keeps ~1e-7 relative
// accuracy even for close pairs.
//
// k_rbf_kernel   K_ij = exp(-|p_i - p_j|^2 / (2 ell^2)) in FP32 (kernel ridge
//                regression systems, Section 3); 64 x 64 tiles of the upper
//                triangle, each stored at both of its places.
// k_rbf_grad_ell out = -sum_ij a_i (dK_ij/d ell) x_j with
//                dK_ij/d ell = K_ij d_ij^2 / ell^3 recomputed per pair, so
//                dK is never formed. Each warp owns a row i; the points and
//                x_j (split into an exact FP32 pair x_hi + x_lo) are staged
//                per chunk in shared memory; per-lane sums are compensated
//                (TwoSum) in FP32 and combined in FP64; a_i multiplies the
//                FP64 row total; the last block sums the block totals in a
//                fixed order.
#include "msp_internal.cuh"

#include <cmath>
#include <mutex>

namespace {

constexpr int kRbfChunk = 1024;

struct PtHL {
    float4 hi, lo;
};

__device__ inline PtHL load_point(const double* __restrict__ P, int64_t i, int dim) {
    float h[4] = {0.f, 0.f, 0.f, 0.f}, l[4] = {0.f, 0.f, 0.f, 0.f};
    for (int d = 0; d < dim; ++d) {
        const double v = P[i * dim + d];
        h[d] = (float)v;
        l[d] = (float)(v - (double)h[d]);
    }
    return {make_float4(h[0], h[1], h[2], h[3]), make_float4(l[0], l[1], l[2], l[3])};
}

__device__ inline float sqdist(const PtHL& a, const PtHL& b) {
    const float dx = (a.hi.x - b.hi.x) + (a.lo.x - b.lo.x);
    const float dy = (a.hi.y - b.hi.y) + (a.lo.y - b.lo.y);
    const float dz = (a.hi.z - b.hi.z) + (a.lo.z - b.lo.z);
    const float dw = (a.hi.w - b.hi.w) + (a.lo.w - b.lo.w);
    return fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, dw * dw)));
}

__device__ inline PtHL zero_point() {
    return {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
}

// One 64 x 64 tile (I, J), I <= J, of the symmetric K per block, written to (I, J)
// and, off the diagonal, transposed to (J, I): a difference and its negative square
// to the same bits, so each pair's distance and expf are formed once. A thread
// forms 4 x 4 entries from point coordinates in registers (6 values of 4 points a
// side at DIM = 3, one 16-byte load each), and a warp covers 32 columns by 16
// rows, so a warp store is 128 bytes of 4 rows one way and 64 bytes of 8 rows the
// other. With every entry formed at its own place, one per thread and step, the
// kernel was bound by issue: 597 us for n = 16384 (1.8 TB/s); now 224 us (4.8 TB/s).
// VEC: rows of K start on 16-byte boundaries. Otherwise the tile goes through
// shared memory (a column of padding: no bank conflicts either way) and is
// stored by words, 128 bytes a warp.
constexpr int kKt = 64;

template <int DIM, bool VEC>
__global__ void __launch_bounds__(256) k_rbf_kernel(const double* __restrict__ P, int64_t n, int nt,
                                                   float inv2l2, float* __restrict__ K, int64_t ldk) {
    __shared__ __align__(16) float ph[2][DIM][kKt], pl[2][DIM][kKt];   // rows' and columns' points, hi and lo
    __shared__ float tile[VEC ? 1 : kKt][VEC ? 1 : kKt + 1];
    // block -> tile of the upper triangle, row by row: start(i) = i nt - i (i - 1) / 2
    const int64_t t = blockIdx.x;
    int I = (int)((2.0f * nt + 1.0f - sqrtf(fmaxf((2.0f * nt + 1.0f) * (2.0f * nt + 1.0f) - 8.0f * (float)t, 0.f))) * 0.5f);
    I = max(0, min(I, nt - 1));
    while (I > 0 && (int64_t)I * nt - (int64_t)I * (I - 1) / 2 > t) --I;
    while (I + 1 < nt && (int64_t)(I + 1) * nt - (int64_t)(I + 1) * I / 2 <= t) ++I;
    const int J = I + (int)(t - ((int64_t)I * nt - (int64_t)I * (I - 1) / 2));
    const int64_t i0 = (int64_t)I * kKt, j0 = (int64_t)J * kKt;
    for (int e = threadIdx.x; e < 2 * kKt * DIM; e += 256) {
        const int side = e / (kKt * DIM), q = (e / DIM) % kKt, d = e % DIM;
        const int64_t i = (side ? j0 : i0) + q;
        const double v = i < n ? P[i * DIM + d] : 0.0;
        const float h = (float)v;
        ph[side][d][q] = h;
        pl[side][d][q] = (float)(v - (double)h);
    }
    __syncthreads();
    // warp w: rows 16 (w & 3) .. + 16, columns 32 (w >> 2) .. + 32
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int r0 = 16 * (w & 3) + 4 * (lane >> 3), c0 = 32 * (w >> 2) + 4 * (lane & 7);
    float s[4][4];
#pragma unroll
    for (int d = DIM - 1; d >= 0; --d) {
        const float4 rh = *reinterpret_cast<const float4*>(&ph[0][d][r0]), rl = *reinterpret_cast<const float4*>(&pl[0][d][r0]);
        const float4 ch = *reinterpret_cast<const float4*>(&ph[1][d][c0]), cl = *reinterpret_cast<const float4*>(&pl[1][d][c0]);
        const float rhv[4] = {rh.x, rh.y, rh.z, rh.w}, rlv[4] = {rl.x, rl.y, rl.z, rl.w};
        const float chv[4] = {ch.x, ch.y, ch.z, ch.w}, clv[4] = {cl.x, cl.y, cl.z, cl.w};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const float dd = (rhv[a] - chv[b]) + (rlv[a] - clv[b]);
                s[a][b] = d == DIM - 1 ? dd * dd : fmaf(dd, dd, s[a][b]);
            }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) s[a][b] = expf(-s[a][b] * inv2l2);
    if constexpr (VEC) {
        const int64_t i = i0 + r0, j = j0 + c0;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            if (i + a >= n) break;
            float* k = K + (i + a) * ldk + j;
            if (j + 3 < n) *reinterpret_cast<float4*>(k) = make_float4(s[a][0], s[a][1], s[a][2], s[a][3]);
            else
#pragma unroll
                for (int b = 0; b < 3; ++b)
                    if (j + b < n) k[b] = s[a][b];
        }
        if (I == J) return;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (j + b >= n) break;
            // the rows' tile is a whole one: J > I
            *reinterpret_cast<float4*>(K + (j + b) * ldk + i) = make_float4(s[0][b], s[1][b], s[2][b], s[3][b]);
        }
    } else {
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) tile[r0 + a][c0 + b] = s[a][b];
        __syncthreads();
        const int c = threadIdx.x & 63;
        for (int r = threadIdx.x >> 6; r < kKt; r += 4)
            if (i0 + r < n && j0 + c < n) K[(i0 + r) * ldk + j0 + c] = tile[r][c];
        if (I == J) return;
        for (int r = threadIdx.x >> 6; r < kKt; r += 4)
            if (j0 + r < n) K[(j0 + r) * ldk + i0 + c] = tile[c][r];
    }
}

template <int DIM>
void launch_rbf_kernel(cudaStream_t st, const double* P, int64_t n, float inv2l2, float* K, int64_t ldk) {
    const int64_t nt = (n + kKt - 1) / kKt;
    const unsigned blocks = (unsigned)(nt * (nt + 1) / 2);
    if (ldk % 4 == 0 && (reinterpret_cast<uintptr_t>(K) & 15) == 0)
        k_rbf_kernel<DIM, true><<<blocks, 256, 0, st>>>(P, n, (int)nt, inv2l2, K, ldk);
    else
        k_rbf_kernel<DIM, false><<<blocks, 256, 0, st>>>(P, n, (int)nt, inv2l2, K, ldk);
}

__device__ inline void two_sum_acc(float& s, float& c, float v) {
    const float t = s + v;
    const float bp = t - s;
    c += (s - (t - bp)) + (v - bp);
    s = t;
}

__global__ void __launch_bounds__(256) k_rbf_grad_ell(const double* __restrict__ P, int64_t n, int dim,
                                                     float inv2l2, const double* __restrict__ a,
                                                     const double* __restrict__ x,
                                                     double* __restrict__ part,
                                                     unsigned int* counter, double* out,
                                                     double scale) {
    __shared__ PtHL pts[kRbfChunk];
    __shared__ float xh[kRbfChunk], xl[kRbfChunk];
    __shared__ double red[8];
    __shared__ bool am_last;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * 8 + w;
    const PtHL pi = (i < n) ? load_point(P, i, dim) : zero_point();
    float s = 0.f, c = 0.f;
    double row = 0.0;
    for (int64_t j0 = 0; j0 < n; j0 += kRbfChunk) {
        const int len = (int)min((int64_t)kRbfChunk, n - j0);
        __syncthreads();
        for (int t = threadIdx.x; t < len; t += blockDim.x) {
            pts[t] = load_point(P, j0 + t, dim);
            const double xv = x[j0 + t];
            const float hi = (float)xv;
            xh[t] = hi;
            xl[t] = (float)(xv - (double)hi);
        }
        __syncthreads();
        if (i < n) {
            for (int t = lane; t < len; t += 32) {
                const float d2 = sqdist(pi, pts[t]);
                const float term = expf(-d2 * inv2l2) * d2;       // K_ij d_ij^2
                const float p = term * xh[t];
                const float e = fmaf(term, xh[t], -p);            // exact product error
                two_sum_acc(s, c, p);
                c += fmaf(term, xl[t], e);
            }
        }
        // fold the chunk into FP64 so the FP32 running sum stays short
        row += (double)s + (double)c;
        s = 0.f;
        c = 0.f;
    }
    row = msp::warp_sum(row);
    double contrib = (lane == 0 && i < n) ? a[i] * row : 0.0;
    if (lane == 0) red[w] = contrib;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int k = 0; k < 8; ++k) tot += red[k];
        part[blockIdx.x] = tot;
        __threadfence();
        const unsigned int tk = atomicAdd(counter, 1u);
        am_last = (tk == gridDim.x - 1);
    }
    __syncthreads();
    if (!am_last || threadIdx.x != 0) return;
    __threadfence();
    double all = 0.0;
    for (unsigned int b = 0; b < gridDim.x; ++b) all += __ldcg(&part[b]);
    *counter = 0;
    *out = -all * scale;
}

// ---------------------------------------------------- no-allocation variant
//
// Scratch of msp_rbf_grad_ell_static: word 0 holds the last-block counter,
// the FP64 block partials start at element 32 (256 bytes in). The grid has
// one block per 8 points, so n is limited to 8 * kStaticMaxBlocks. Every GPU
// that loads the library holds this array (about 512 KiB) until exit.
constexpr int64_t kStaticMaxBlocks = 65536;
constexpr int64_t kStaticMaxN = 8 * kStaticMaxBlocks;
static __device__ __align__(256) double g_rbf_grad_static[32 + kStaticMaxBlocks];

std::mutex g_static_mu;
double* g_static_ptr[64] = {};   // device address of the array, per device

}  // namespace

extern "C" {

msp_status msp_rbf_grad_ell_static(const double* points, int64_t n, int dim, double ell,
                                   const double* a, const double* x, double* out, void* stream) {
    if (!points || !a || !x || !out || n < 1 || dim < 1 || dim > 4 || !(ell > 0.0))
        return msp_set_error(nullptr, MSP_EINVAL,
                             "rbf_grad_ell_static: need n >= 1, 1 <= dim <= 4, ell > 0, non-NULL arrays");
    if (n > kStaticMaxN)
        return msp_set_error(nullptr, MSP_EINVAL,
                             "rbf_grad_ell_static: n = %lld exceeds the static scratch limit n <= %lld",
                             (long long)n, (long long)kStaticMaxN);
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return msp_set_error(nullptr, MSP_ECUDA, "rbf_grad_ell_static: no current CUDA device");
    }
    cudaStream_t st = (cudaStream_t)stream;
    if (st) {
        int sdev = -1;
        if (cudaStreamGetDevice(st, &sdev) != cudaSuccess || sdev != dev) {
            cudaGetLastError();
            return msp_set_error(nullptr, MSP_EINVAL,
                                 "rbf_grad_ell_static: the stream does not belong to the current device %d", dev);
        }
    }
    double* scratch = nullptr;
    {
        // set-up, once per device, with that device current: the host-side
        // name of the array is not a device address
        std::lock_guard<std::mutex> lock(g_static_mu);
        if (!g_static_ptr[dev]) {
            void* p = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&p, g_rbf_grad_static);
            if (e != cudaSuccess || !p) {
                cudaGetLastError();
                return msp_set_error(nullptr, MSP_ECUDA, "rbf_grad_ell_static: cudaGetSymbolAddress: %s",
                                     cudaGetErrorString(e));
            }
            g_static_ptr[dev] = (double*)p;
        }
        scratch = g_static_ptr[dev];
    }
    unsigned int* counter = reinterpret_cast<unsigned int*>(scratch);
    // the counter must start at zero (the array keeps the last call's contents)
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned int), st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return msp_set_error(nullptr, MSP_ECUDA, "rbf_grad_ell_static: %s", cudaGetErrorString(e));
    }
    const unsigned blocks = (unsigned)((n + 7) / 8);
    k_rbf_grad_ell<<<blocks, 256, 0, st>>>(points, n, dim, (float)(1.0 / (2.0 * ell * ell)), a, x,
                                           scratch + 32, counter, out, 1.0 / (ell * ell * ell));
    e = cudaGetLastError();
    if (e != cudaSuccess)
        return msp_set_error(nullptr, MSP_ECUDA, "rbf_grad_ell_static: launch: %s", cudaGetErrorString(e));
    return MSP_OK;
}

msp_status msp_rbf_kernel(msp_ctx* ctx, const double* points, int64_t n, int dim, double ell,
                          float* K, int64_t ldk) {
    if (!ctx) return msp_set_error(nullptr, MSP_EINVAL, "ctx is NULL");
    if (!points || !K || n < 1 || ldk < n || dim < 1 || dim > 4 || !(ell > 0.0))
        return msp_set_error(ctx, MSP_EINVAL, "rbf_kernel: need n >= 1, 1 <= dim <= 4, ell > 0, ldk >= n");
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != ctx->device) cudaSetDevice(ctx->device);
    const float inv2l2 = (float)(1.0 / (2.0 * ell * ell));
    switch (dim) {
        case 1: launch_rbf_kernel<1>(ctx->stream, points, n, inv2l2, K, ldk); break;
        case 2: launch_rbf_kernel<2>(ctx->stream, points, n, inv2l2, K, ldk); break;
        case 3: launch_rbf_kernel<3>(ctx->stream, points, n, inv2l2, K, ldk); break;
        default: launch_rbf_kernel<4>(ctx->stream, points, n, inv2l2, K, ldk); break;
    }
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

msp_status msp_rbf_grad_ell(msp_ctx* ctx, const double* points, int64_t n, int dim, double ell,
                            const double* a, const double* x, double* out) {
    if (!ctx) return msp_set_error(nullptr, MSP_EINVAL, "ctx is NULL");
    if (!points || !a || !x || !out || n < 1 || dim < 1 || dim > 4 || !(ell > 0.0))
        return msp_set_error(ctx, MSP_EINVAL, "rbf_grad_ell: need n >= 1, 1 <= dim <= 4, ell > 0");
    msp::DeviceGuard guard(ctx->device);
    const unsigned blocks = (unsigned)((n + 7) / 8);
    void* scr = nullptr;
    MSP_TRY(msp_scratch(ctx, (size_t)blocks * 8 + 256, &scr));
    CtlBlock* ctl = (CtlBlock*)ctx->ctl;
    k_rbf_grad_ell<<<blocks, 256, 0, ctx->stream>>>(points, n, dim, (float)(1.0 / (2.0 * ell * ell)), a,
                                                    x, (double*)scr, &ctl->last_block_counter, out,
                                                    1.0 / (ell * ell * ell));
    MSP_CHECK_LAUNCH(ctx);
    return MSP_OK;
}

}  // extern "C"
