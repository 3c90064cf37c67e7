// Kernels of the nested-projection stage (Sec. 3.1, Eq. nested_proj): the
// staggered divergence and gradient of Sec. 2.1 on block sets, the marker
// residual and the two dense products with the factors of the force Schur
// complement's inverse (Sec. 3.2).  The stage itself is composed in
// lgf_capi.cu from these and the Poisson, integrating-factor and IB passes.
//
// Cell n holds face k at (n + (1 - e_k)/2) dx, so
//   (Dbar u)(n) = sum_k [u_k(n + e_k) - u_k(n)] / dx     faces -> cells
//   (G q)_k(n)  = [q(n) - q(n - e_k)] / dx               cells -> faces
// and G^dagger = -Dbar.  Both read the block itself and, where the shift
// leaves it, the neighbour block of a CurlPlan (dir +1 for Dbar, -1 for G);
// values outside the input block set are zero.  A thread makes 16 bytes of a row of
// outputs.
#include <algorithm>
#include <cstring>

#include "lgf_async.cuh"
#include "lgf_internal.cuh"

namespace lgf {
namespace {

// Both stencils take 16 bytes of a row (VN cells) per thread: vector loads of
// the cells and of the rows shifted along y and z, and one more value (or the
// neighbour block's) for the shift along x.  One cell per thread left them bound by
// the latency of their 4-byte loads: 19 and 21 us, now 16 each, where 556 blocks of
// 16^3 move 36 and 64 MB; the arithmetic of a cell is unchanged.  VEC = false: one cell per thread,
// for fields off the 16-byte alignment.
// out(n) = scale * sum_k [(a - c)_k(n + e_k) - (a - c)_k(n)]   (c may be null)
template <typename T, int LB, bool VEC>
__global__ void __launch_bounds__(256) k_div(const T *__restrict__ a, const T *__restrict__ c, T *__restrict__ out,
                                             const int *__restrict__ nbr, int64_t ncell, int64_t in_c, T scale)
{
    using VT = typename CellVec<T, VEC>::V;
    constexpr int VN = sizeof(VT) / sizeof(T);
    const int64_t idx = (blockIdx.x * 256LL + threadIdx.x) * VN;
    if (idx >= ncell) return;
    constexpr int b = 1 << LB, bm = b - 1;
    const int o = (int)(idx >> (3 * LB));
    const int loc = (int)(idx & ((1LL << (3 * LB)) - 1));
    const int cc[3] = {loc & bm, (loc >> LB) & bm, loc >> (2 * LB)};
    const int *nb = nbr + 4 * (int64_t)o;
    // VN cells of component k from element i of block blk (absent: zero)
    auto vec = [&](int k, int blk, int l, T (&v)[VN]) {
        VT r = VT{};
        if (blk >= 0) {
            const int64_t i = k * in_c + ((int64_t)blk << (3 * LB)) + l;
            r = *reinterpret_cast<const VT *>(a + i);
            if (c) {
                const VT q = *reinterpret_cast<const VT *>(c + i);
                const T *qs = reinterpret_cast<const T *>(&q);
                T *rs = reinterpret_cast<T *>(&r);
#pragma unroll
                for (int e = 0; e < VN; ++e) rs[e] -= qs[e];
            }
        }
        const T *rs = reinterpret_cast<const T *>(&r);
#pragma unroll
        for (int e = 0; e < VN; ++e) v[e] = rs[e];
    };
    T s[VN];
#pragma unroll
    for (int e = 0; e < VN; ++e) s[e] = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        T self[VN], next[VN];
        vec(k, nb[0], loc, self);
        if (k == 0) {
            const bool edge = cc[0] + VN > bm;
            const int blk = edge ? nb[1] : nb[0];
            T last = T(0);
            if (blk >= 0) {
                const int64_t i = ((int64_t)blk << (3 * LB)) + (edge ? loc - cc[0] : loc + VN);
                last = c ? a[i] - c[i] : a[i];
            }
#pragma unroll
            for (int e = 0; e < VN; ++e) next[e] = e + 1 < VN ? self[e + 1] : last;
        } else {
            const int step = 1 << (k * LB);   // along y or z
            const bool edge = cc[k] == bm;
            vec(k, edge ? nb[1 + k] : nb[0], edge ? loc - bm * step : loc + step, next);
        }
#pragma unroll
        for (int e = 0; e < VN; ++e) s[e] += next[e] - self[e];
    }
    VT r;
    T *rs = reinterpret_cast<T *>(&r);
#pragma unroll
    for (int e = 0; e < VN; ++e) rs[e] = scale * s[e];
    *reinterpret_cast<VT *>(out + idx) = r;
}

// out_k(n) = a_k(n) - inv_dx * [d(n) - d(n - e_k)] - c_k(n)   (c may be null);
// d on the plan's source blocks, a, c, out on its target blocks.
template <typename T, int LB, bool VEC>
__global__ void __launch_bounds__(256) k_grad_combine(const T *__restrict__ d, const T *__restrict__ a,
                                                      const T *__restrict__ c, T *__restrict__ out,
                                                      const int *__restrict__ nbr, int64_t ncell, T inv_dx)
{
    using VT = typename CellVec<T, VEC>::V;
    constexpr int VN = sizeof(VT) / sizeof(T);
    const int64_t idx = (blockIdx.x * 256LL + threadIdx.x) * VN;
    if (idx >= ncell) return;
    constexpr int b = 1 << LB, bm = b - 1;
    const int o = (int)(idx >> (3 * LB));
    const int loc = (int)(idx & ((1LL << (3 * LB)) - 1));
    const int cc[3] = {loc & bm, (loc >> LB) & bm, loc >> (2 * LB)};
    const int *nb = nbr + 4 * (int64_t)o;
    auto vec = [&](int blk, int l, T (&v)[VN]) {
        const VT r = blk >= 0 ? *reinterpret_cast<const VT *>(d + ((int64_t)blk << (3 * LB)) + l) : VT{};
        const T *rs = reinterpret_cast<const T *>(&r);
#pragma unroll
        for (int e = 0; e < VN; ++e) v[e] = rs[e];
    };
    T dn[VN];
    vec(nb[0], loc, dn);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        T dm[VN];
        if (k == 0) {
            const bool edge = cc[0] == 0;
            const int blk = edge ? nb[1] : nb[0];
            dm[0] = blk >= 0 ? d[((int64_t)blk << (3 * LB)) + (edge ? loc + bm : loc - 1)] : T(0);
#pragma unroll
            for (int e = 1; e < VN; ++e) dm[e] = dn[e - 1];
        } else {
            const int step = 1 << (k * LB);
            const bool edge = cc[k] == 0;
            vec(edge ? nb[1 + k] : nb[0], edge ? loc + bm * step : loc - step, dm);
        }
        const int64_t i = k * ncell + idx;
        VT av = *reinterpret_cast<const VT *>(a + i), cv = VT{};
        if (c) cv = *reinterpret_cast<const VT *>(c + i);
        T *as = reinterpret_cast<T *>(&av);
        const T *cs = reinterpret_cast<const T *>(&cv);
#pragma unroll
        for (int e = 0; e < VN; ++e) {
            T v = as[e] - inv_dx * (dn[e] - dm[e]);
            if (c) v -= cs[e];
            as[e] = v;
        }
        *reinterpret_cast<VT *>(out + i) = av;
    }
}

template <typename T>
__global__ void k_sub(const T *__restrict__ x, const T *__restrict__ y, T *__restrict__ out, int64_t n)
{
    const int64_t i = blockIdx.x * 256LL + threadIdx.x;
    if (i < n) out[i] = x[i] - y[i];
}

// y = W x, W row-major n x n: one warp per row, lanes stride the row
// (coalesced), shuffle reduction.
template <typename T>
__global__ void __launch_bounds__(256) k_gemv_n(const T *__restrict__ W, const T *__restrict__ x, T *__restrict__ y,
                                                int n)
{
    const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= n) return;
    const T *w = W + (int64_t)row * n;
    T s = T(0);
    for (int j = lane; j < n; j += 32) s += w[j] * x[j];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if (lane == 0) y[row] = s;
}

// y = W^T x: a CTA owns 32 columns; its 8 warps sum rows i = g (mod 8) with
// lane = column (each warp reads 32 contiguous values of a row), then the 8
// partial sums are added in shared memory.
template <typename T>
__global__ void __launch_bounds__(256) k_gemv_t(const T *__restrict__ W, const T *__restrict__ x, T *__restrict__ y,
                                                int n)
{
    __shared__ T part[8][32];
    const int col = blockIdx.x * 32 + (threadIdx.x & 31);
    const int g = threadIdx.x >> 5;
    T s = T(0);
    if (col < n)
        for (int i = g; i < n; i += 8) s += W[(int64_t)i * n + col] * x[i];
    part[g][threadIdx.x & 31] = s;
    __syncthreads();
    if (g == 0 && col < n) {
        T t = T(0);
#pragma unroll
        for (int q = 0; q < 8; ++q) t += part[q][threadIdx.x];
        y[col] = t;
    }
}

// f = W^T (W x), x = U - ub, in one pass over W (n x n, row-major), which two
// products read twice: HBM bounds both (15360^2 in FP32 is 944 MB, 139 us at
// the measured copy bandwidth; two products took 450 us, one pass takes 172).
// A CTA of 512 threads holds a whole row
// in registers (NK 16-byte vectors per thread, the vectors of a warp
// contiguous), forms y_r = W_r x, and adds y_r W_r to its own sum of W^T y, also in
// registers; the next row is in flight meanwhile.  One barrier per row (the
// partial sums of the warps alternate between two buffers).  CTA g's sum goes to
// part[g], added in a fixed order by k_part_sum.  Rows go round robin to one
// CTA per SM.  VEC: 16-byte loads (n a multiple of the vector, W aligned).
constexpr int kGramThreads = 512;
template <typename T>
struct GramVec;
template <>
struct GramVec<float> {
    using V = float4;
};
template <>
struct GramVec<double> {
    using V = double2;
};
template <typename T, int NK, bool VEC>
__global__ void __launch_bounds__(kGramThreads, 1) k_gram(const T *__restrict__ W, const T *__restrict__ U,
                                                          const T *__restrict__ ub, T *__restrict__ part, int n)
{
    using VT = typename GramVec<T>::V;
    constexpr int NV = sizeof(VT) / sizeof(T), NT = kGramThreads, NW = NT / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *xs = reinterpret_cast<T *>(smem_raw);   // [NK * NT * NV], zero past n
    __shared__ T red[2][NW];
    const int tid = threadIdx.x;
    for (int i = tid; i < NK * NT * NV; i += NT) xs[i] = i < n ? U[i] - ub[i] : T(0);
    __syncthreads();
    auto load = [&](T (&a)[NK][NV], int row) {
        const T *w = W + (int64_t)row * n;
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            const int c = (k * NT + tid) * NV;
            if constexpr (VEC) {
                const VT v = c < n ? __ldcs(reinterpret_cast<const VT *>(w + c)) : VT{};
                memcpy(a[k], &v, sizeof(VT));
            } else {
#pragma unroll
                for (int e = 0; e < NV; ++e) a[k][e] = c + e < n ? w[c + e] : T(0);
            }
        }
    };
    T acc[NK][NV], cur[NK][NV], nxt[NK][NV];
#pragma unroll
    for (int k = 0; k < NK; ++k)
#pragma unroll
        for (int e = 0; e < NV; ++e) acc[k][e] = T(0);
    auto row_step = [&](const T (&a)[NK][NV], int buf) {
        T s = T(0);
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            const VT xv = *reinterpret_cast<const VT *>(xs + (k * NT + tid) * NV);
            const T *x = reinterpret_cast<const T *>(&xv);
#pragma unroll
            for (int e = 0; e < NV; ++e) s += a[k][e] * x[e];
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if ((tid & 31) == 0) red[buf][tid >> 5] = s;
        __syncthreads();
        T y = T(0);
#pragma unroll
        for (int q = 0; q < NW; ++q) y += red[buf][q];
#pragma unroll
        for (int k = 0; k < NK; ++k)
#pragma unroll
            for (int e = 0; e < NV; ++e) acc[k][e] += y * a[k][e];
    };
    const int g = gridDim.x;
    int r = blockIdx.x;   // gridDim.x <= n
    load(cur, r);
    for (; r < n; r += 2 * g) {
        if (r + g < n) load(nxt, r + g);
        row_step(cur, 0);
        if (r + g >= n) break;   // uniform over the CTA
        if (r + 2 * g < n) load(cur, r + 2 * g);
        row_step(nxt, 1);
    }
    T *o = part + (int64_t)blockIdx.x * n;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        const int c = (k * NT + tid) * NV;
#pragma unroll
        for (int e = 0; e < NV; ++e)
            if (c + e < n) o[c + e] = acc[k][e];
    }
}

// y = sum of the m rows of part (m x n): k_gemv_t's split with unit weights.
template <typename T>
__global__ void __launch_bounds__(256) k_part_sum(const T *__restrict__ part, T *__restrict__ y, int m, int n)
{
    __shared__ T sum[8][32];
    const int col = blockIdx.x * 32 + (threadIdx.x & 31);
    const int g = threadIdx.x >> 5;
    T s = T(0);
    if (col < n)
        for (int i = g; i < m; i += 8) s += part[(int64_t)i * n + col];
    sum[g][threadIdx.x & 31] = s;
    __syncthreads();
    if (g == 0 && col < n) {
        T t = T(0);
#pragma unroll
        for (int q = 0; q < 8; ++q) t += sum[q][threadIdx.x];
        y[col] = t;
    }
}

template <typename T, int NK, bool VEC>
lgf_status launch_gram_k(lgf_ctx *ctx, const T *W, const T *U, const T *ub, T *part, T *fh, int n, int grid,
                         cudaStream_t s)
{
    constexpr size_t smem = (size_t)NK * kGramThreads * 16;
    auto kern = k_gram<T, NK, VEC>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaFuncSetAttribute");
    }
    kern<<<grid, kGramThreads, smem, s>>>(W, U, ub, part, n);
    k_part_sum<T><<<(n + 31) / 32, 256, 0, s>>>(part, fh, grid, n);
    return LGF_OK;
}

// The row length a thread's NK vectors cover picks NK: 1, 2, 4 or 8.
template <typename T, bool VEC>
lgf_status launch_gram(lgf_ctx *ctx, const T *W, const T *U, const T *ub, T *part, T *fh, int n, int grid,
                       cudaStream_t s)
{
    constexpr int per = kGramThreads * (16 / (int)sizeof(T));
    if (n <= per) return launch_gram_k<T, 1, VEC>(ctx, W, U, ub, part, fh, n, grid, s);
    if (n <= 2 * per) return launch_gram_k<T, 2, VEC>(ctx, W, U, ub, part, fh, n, grid, s);
    if (n <= 4 * per) return launch_gram_k<T, 4, VEC>(ctx, W, U, ub, part, fh, n, grid, s);
    return launch_gram_k<T, 8, VEC>(ctx, W, U, ub, part, fh, n, grid, s);
}

template <typename T>
lgf_status gram(lgf_ctx *ctx, const void *W, const void *U, const void *ub, void *part, void *fh, int n, int grid,
                cudaStream_t s)
{
    const bool vec = n % (16 / (int)sizeof(T)) == 0 && reinterpret_cast<uintptr_t>(W) % 16 == 0;
    return vec ? launch_gram<T, true>(ctx, (const T *)W, (const T *)U, (const T *)ub, (T *)part, (T *)fh, n, grid, s)
               : launch_gram<T, false>(ctx, (const T *)W, (const T *)U, (const T *)ub, (T *)part, (T *)fh, n, grid, s);
}

// CTAs of the one-pass product (0: rows too long for a CTA's registers).
int gram_grid(const lgf_ctx *ctx, int n)
{
    const int most = 8 * kGramThreads * (ctx->prec == LGF_F64 ? 2 : 4);   // 16384 in FP32, 8192 in FP64
    int nsm = 0;
    if (n > most || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess) return 0;
    return std::min(n, nsm);
}

template <typename T, int LB>
void launch_div_lb(cudaStream_t s, const T *a, const T *c, T *out, const int *nbr, int64_t ncell,
                   int64_t in_c, T scale)
{
    if (cells_aligned(a, c, out))
        k_div<T, LB, true><<<cell_grid<T, true>(ncell), 256, 0, s>>>(a, c, out, nbr, ncell, in_c, scale);
    else
        k_div<T, LB, false><<<cell_grid<T, false>(ncell), 256, 0, s>>>(a, c, out, nbr, ncell, in_c, scale);
}

template <typename T, int LB>
void launch_grad_lb(cudaStream_t s, const T *d, const T *a, const T *c, T *out, const int *nbr,
                    int64_t ncell, T inv_dx)
{
    if (cells_aligned(d, a, out) && cells_aligned(c, nullptr, nullptr))
        k_grad_combine<T, LB, true><<<cell_grid<T, true>(ncell), 256, 0, s>>>(d, a, c, out, nbr, ncell, inv_dx);
    else
        k_grad_combine<T, LB, false><<<cell_grid<T, false>(ncell), 256, 0, s>>>(d, a, c, out, nbr, ncell, inv_dx);
}

template <typename T>
lgf_status div_t(lgf_ctx *ctx, int lb, const T *a, const T *c, T *out, const int *nbr, int64_t ncell, int64_t in_c,
                 T scale, cudaStream_t s)
{
    const int ph = prof_begin(ctx, s, "stage_div");
    switch (lb) {
    case 2: launch_div_lb<T, 2>(s, a, c, out, nbr, ncell, in_c, scale); break;
    case 3: launch_div_lb<T, 3>(s, a, c, out, nbr, ncell, in_c, scale); break;
    case 4: launch_div_lb<T, 4>(s, a, c, out, nbr, ncell, in_c, scale); break;
    case 5: launch_div_lb<T, 5>(s, a, c, out, nbr, ncell, in_c, scale); break;
    case 6: launch_div_lb<T, 6>(s, a, c, out, nbr, ncell, in_c, scale); break;
    default: return fail(ctx, LGF_EINVAL, "stage: block edge must be 4..64");
    }
    LGF_CHECK_LAUNCH(ctx, "stage divergence");
    prof_end(ctx, s, ph);
    return LGF_OK;
}

template <typename T>
lgf_status grad_t(lgf_ctx *ctx, int lb, const T *d, const T *a, const T *c, T *out, const int *nbr, int64_t ncell,
                  T inv_dx, cudaStream_t s)
{
    const int ph = prof_begin(ctx, s, "stage_grad");
    switch (lb) {
    case 2: launch_grad_lb<T, 2>(s, d, a, c, out, nbr, ncell, inv_dx); break;
    case 3: launch_grad_lb<T, 3>(s, d, a, c, out, nbr, ncell, inv_dx); break;
    case 4: launch_grad_lb<T, 4>(s, d, a, c, out, nbr, ncell, inv_dx); break;
    case 5: launch_grad_lb<T, 5>(s, d, a, c, out, nbr, ncell, inv_dx); break;
    case 6: launch_grad_lb<T, 6>(s, d, a, c, out, nbr, ncell, inv_dx); break;
    default: return fail(ctx, LGF_EINVAL, "stage: block edge must be 4..64");
    }
    LGF_CHECK_LAUNCH(ctx, "stage gradient");
    prof_end(ctx, s, ph);
    return LGF_OK;
}

// The timeout path of the bounded waits: an mbarrier expecting one arrival
// that never comes (no thread arrives, no copy is issued), so the wait runs
// out after `cycles` and sets the error word.
__global__ void k_wait_selftest(int *err, long long cycles)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) async::mbar_init(&bar);
    __syncthreads();
    async::mbar_wait(&bar, 0, err, cycles);
}

int lb_of(int b)
{
    int l = 0;
    while ((1 << l) < b) ++l;
    return (1 << l) == b ? l : -1;
}

}  // namespace

// out = (1/dx) Dbar (a - c) on the plan's target blocks (plan dir +1; a, c on
// its source blocks, c may be null).
lgf_status stage_div(lgf_ctx *ctx, const CurlPlan *pl, const void *a, const void *c, void *out, double dx,
                     cudaStream_t s)
{
    const int64_t b3 = (int64_t)pl->b * pl->b * pl->b;
    const int64_t ncell = (int64_t)(pl->tgt.size() / 3) * b3, in_c = (int64_t)(pl->src.size() / 3) * b3;
    if (ncell == 0) return LGF_OK;
    if (ctx->prec == LGF_F64)
        return div_t<double>(ctx, lb_of(pl->b), (const double *)a, (const double *)c, (double *)out, pl->nbr_dev,
                             ncell, in_c, 1.0 / dx, s);
    return div_t<float>(ctx, lb_of(pl->b), (const float *)a, (const float *)c, (float *)out, pl->nbr_dev, ncell, in_c,
                        (float)(1.0 / dx), s);
}

// out = a - G d - c on the plan's target blocks (plan dir -1; d on its source
// blocks; a, c, out three components on its target blocks, c may be null).
lgf_status stage_grad(lgf_ctx *ctx, const CurlPlan *pl, const void *d, const void *a, const void *c, void *out,
                      double dx, cudaStream_t s)
{
    const int64_t b3 = (int64_t)pl->b * pl->b * pl->b;
    const int64_t ncell = (int64_t)(pl->tgt.size() / 3) * b3;
    if (ncell == 0) return LGF_OK;
    if (ctx->prec == LGF_F64)
        return grad_t<double>(ctx, lb_of(pl->b), (const double *)d, (const double *)a, (const double *)c,
                              (double *)out, pl->nbr_dev, ncell, 1.0 / dx, s);
    return grad_t<float>(ctx, lb_of(pl->b), (const float *)d, (const float *)a, (const float *)c, (float *)out,
                         pl->nbr_dev, ncell, (float)(1.0 / dx), s);
}

lgf_status wait_selftest(lgf_ctx *ctx, long long cycles, cudaStream_t s)
{
    k_wait_selftest<<<1, 32, 0, s>>>(ctx->err_dev, cycles);
    LGF_CHECK_LAUNCH(ctx, "wait self-test");
    return LGF_OK;
}

size_t stage_force_scratch(const lgf_ctx *ctx, const void *W2, int n)
{
    return W2 ? 0 : (size_t)gram_grid(ctx, n) * n * (ctx->prec == LGF_F64 ? 8 : 4);
}

// rhs = U - ub; y = W1 rhs; fh = W2 y (W2 null: W1^T y).  Vectors of n values.
// W2 null and rows that fit a CTA's registers: both products in one pass over
// W1 (k_gram; part as sized by stage_force_scratch, rhs and y unused).  On
// 15360^2 FP32 the two products took 450 us.
lgf_status stage_force(lgf_ctx *ctx, const void *U, const void *ub, const void *W1, const void *W2, void *rhs, void *y,
                       void *fh, void *part, int n, cudaStream_t s)
{
    if (n == 0) return LGF_OK;
    if (const int grid = W2 ? 0 : gram_grid(ctx, n)) {
        const int ph = prof_begin(ctx, s, "stage_force");
        const lgf_status st = ctx->prec == LGF_F64 ? gram<double>(ctx, W1, U, ub, part, fh, n, grid, s)
                                                   : gram<float>(ctx, W1, U, ub, part, fh, n, grid, s);
        if (st != LGF_OK) return st;
        LGF_CHECK_LAUNCH(ctx, "stage force solve");
        prof_end(ctx, s, ph);
        return LGF_OK;
    }
    const unsigned gv = (unsigned)((n + 255) / 256), gn = (unsigned)((n + 7) / 8), gt = (unsigned)((n + 31) / 32);
    const int ph = prof_begin(ctx, s, "stage_force");
    if (ctx->prec == LGF_F64) {
        k_sub<double><<<gv, 256, 0, s>>>((const double *)U, (const double *)ub, (double *)rhs, n);
        k_gemv_n<double><<<gn, 256, 0, s>>>((const double *)W1, (const double *)rhs, (double *)y, n);
        if (W2)
            k_gemv_n<double><<<gn, 256, 0, s>>>((const double *)W2, (const double *)y, (double *)fh, n);
        else
            k_gemv_t<double><<<gt, 256, 0, s>>>((const double *)W1, (const double *)y, (double *)fh, n);
    } else {
        k_sub<float><<<gv, 256, 0, s>>>((const float *)U, (const float *)ub, (float *)rhs, n);
        k_gemv_n<float><<<gn, 256, 0, s>>>((const float *)W1, (const float *)rhs, (float *)y, n);
        if (W2)
            k_gemv_n<float><<<gn, 256, 0, s>>>((const float *)W2, (const float *)y, (float *)fh, n);
        else
            k_gemv_t<float><<<gt, 256, 0, s>>>((const float *)W1, (const float *)y, (float *)fh, n);
    }
    LGF_CHECK_LAUNCH(ctx, "stage force solve");
    prof_end(ctx, s, ph);
    return LGF_OK;
}

}  // namespace lgf
