// prep.cu -- the small kernels around the distance kernels:
//   maxabs      max |x| over a stage's data (fixed-point scale, finiteness check)
//   qsum        exact sum of s^2 over a stage's coordinates, s = round(x 2^F)
//               (the integer that J is formed from, Eq. 3)
//   gather      X_s = rows of X at the subset indices (Algorithm: the per% subset)
//   init        initial centers = chosen points of X_s (Algorithm: random initial centers)
//   stage_begin fixed-point scales and loop state of one stage, zero sums, FP32 /
//               transposed copies of the FP64 centers and ||c||^2
//   finalize    new centers = cluster means (Lloyd's method, Section 4.1), the
//               largest movement (stop test, Sections 5-6), J (Eq. 3)
//   recheck     FP64 re-evaluation of near-tie points (ties -> lowest index)
#include <algorithm>
#include <cfloat>
#include <cstdint>

#include "api_internal.h"
#include "stage_dev.cuh"

namespace km2 {

namespace {

__device__ __forceinline__ unsigned int abs_bits(float v)
{
    return __float_as_uint(v) & 0x7fffffffu;   // NaN keeps a payload above +inf
}

__device__ __forceinline__ unsigned int warp_max_u32(unsigned int v)
{
    for (int o = 16; o; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Block-wide maximum into st->maxabs_bits: one atomic per block.
__device__ __forceinline__ void block_max_to(unsigned int m, StageState* st)
{
    __shared__ unsigned int wm[32];
    m = warp_max_u32(m);
    if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = threadIdx.x < (blockDim.x >> 5) ? wm[threadIdx.x] : 0u;
        m = warp_max_u32(m);
        if (threadIdx.x == 0 && m) atomicMax(&st->maxabs_bits, m);
    }
}

__global__ void maxabs_kernel(const float* __restrict__ X, long long count, int vec4,
                              StageState* st)
{
    unsigned int m = 0;
    long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long stride = (long long)gridDim.x * blockDim.x;
    long long done = 0;
    if (vec4) {
        const float4* X4 = reinterpret_cast<const float4*>(X);
        long long n4 = count >> 2;
#pragma unroll 4
        for (long long i = tid; i < n4; i += stride) {
            float4 v = __ldg(X4 + i);
            m = max(m, max(max(abs_bits(v.x), abs_bits(v.y)), max(abs_bits(v.z), abs_bits(v.w))));
        }
        done = n4 << 2;
    }
    for (long long i = done + tid; i < count; i += stride) m = max(m, abs_bits(__ldg(X + i)));
    block_max_to(m, st);
}

// Exact sum of s^2 over count coordinates (the same integers the cluster sums
// add), into st->q.  Memory-bound: ~9 instructions per coordinate (one 128-bit
// product and sum per coordinate took 2.5x the time of reading X; n = 5e5, d =
// 128: 125 us).
__global__ void qsum_kernel(const float* __restrict__ X, long long count, int vec4,
                            StageState* st)
{
    __shared__ unsigned long long wl[8], wh[8];
    if (st->error) return;
    const float scale = st->scaleF;
    QSum q;
    long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long stride = (long long)gridDim.x * blockDim.x;
    long long done = 0;
    if (vec4) {
        const float4* X4 = reinterpret_cast<const float4*>(X);
        long long n4 = count >> 2;
        for (long long i = tid; i < n4;) {
            const long long end = min(n4, i + stride * (1 << 14));   // 2^16 coordinates
#pragma unroll 4
            for (; i < end; i += stride) {
                const float4 v = __ldg(X4 + i);
                q.add(v.x, scale);
                q.add(v.y, scale);
                q.add(v.z, scale);
                q.add(v.w, scale);
            }
            q.fold();
        }
        done = n4 << 2;
    }
    int left = 1 << 16;
    for (long long i = done + tid; i < count; i += stride) {
        q.add(__ldg(X + i), scale);
        if (--left == 0) { q.fold(); left = 1 << 16; }
    }
    q.fold();
    unsigned __int128 a = warp_sum_u128(q.total);
    if ((threadIdx.x & 31) == 0) {
        wl[threadIdx.x >> 5] = (unsigned long long)a;
        wh[threadIdx.x >> 5] = (unsigned long long)(a >> 64);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a += ((unsigned __int128)wh[w] << 64) | wl[w];
        if (a) wide_add4(st->q, a);
    }
}

__global__ void gather_kernel(const float* __restrict__ X, int d,
                              const long long* __restrict__ subset, long long m,
                              float* __restrict__ Xs, StageState* st)
{
    unsigned int mx = 0;
    long long total = m * (long long)d;
    long long stride = (long long)gridDim.x * blockDim.x;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += stride) {
        long long p = e / d;
        int t = (int)(e - p * d);
        float v = X[subset[p] * (long long)d + t];
        Xs[e] = v;
        mx = max(mx, abs_bits(v));
    }
    block_max_to(mx, st);
}

__global__ void init_centers_kernel(const float* __restrict__ Xs, int d,
                                    const long long* __restrict__ pos, int k,
                                    double* __restrict__ c64)
{
    long long total = (long long)k * d;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        long long j = e / d;
        int t = (int)(e - j * d);
        c64[e] = (double)Xs[pos[j] * (long long)d + t];
    }
}

// Start of a stage (st zeroed, maxabs_bits set): loop state and scales, zero
// sums and counts, the centers' FP32 copies (padding: zeros in c32t, the largest
// finite float in cnorm, so that packing an index into its low mantissa bits
// never makes a NaN and it never wins or ties), ||c_j||^2 and their maximum,
// rounded up.  One warp per center over many CTAs (one CTA for all centers took
// 149 us at k = 1024, d = 128), and one launch where three memsets, two fills and
// two kernels did it.
__global__ void __launch_bounds__(256) stage_begin_kernel(Centers c, Accum acc, StageState* st,
                                                          double tol, int max_iter, long long cn_len)
{
    const long long gt = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (gt == 0) stage_init_dev(st, c.d, tol, max_iter);
    const long long kd = (long long)c.k * c.d;
    for (long long e = gt; e < kd; e += stride) { acc.s_lo[e] = 0; acc.s_hi[e] = 0; }
    for (long long e = gt; e < c.k; e += stride) acc.cnt[e] = 0;
    for (long long e = c.k + gt; e < cn_len; e += stride) c.cnorm[e] = FLT_MAX;
    const long long tot = (long long)c.dpad * c.kpad;
    for (long long e = gt; e < tot; e += stride) {
        const int t = (int)(e / c.kpad), j = (int)(e - (long long)t * c.kpad);
        if (t >= c.d || j >= c.k) c.c32t[e] = 0.0f;
    }
    const int lane = threadIdx.x & 31;
    double mx = 0.0;
    for (long long j = gt >> 5; j < c.k; j += stride >> 5) {
        double nn = 0.0;
        for (int t = lane; t < c.d; t += 32) {
            const double v = c.c64[j * c.d + t];
            nn = fma(v, v, nn);
            c.c32[j * c.d + t] = (float)v;
            c.c32t[(long long)t * c.kpad + j] = (float)v;
        }
        nn = warp_sum_f64(nn);
        if (lane == 0) c.cnorm[j] = (float)nn;
        mx = fmax(mx, nn);
    }
    // non-negative floats order as their bits; rounding up keeps the order
    if (lane == 0 && mx > 0.0)
        atomicMax(reinterpret_cast<unsigned int*>(&st->cmax2), __float_as_uint(__double2float_ru(mx)));
}

// New centers (one warp each) and their divisions (one thread each), then, in the
// CTA that finishes last, movement, J and loop control for the next iteration.
// What bounds it: FP64, ~60 instructions per center and 32 coordinates, each 16
// cycles of its SM's pipe.  So the centers are dealt out over the SMs one warp at a
// time, and the CTA's divisions run as one warp's instructions.  One CTA with the
// compiler's 128-bit division, one lane and center after the other: 51 us for k =
// 50, d = 5, 134 us for k = 100, d = 37; with 8 centers per CTA and the divisions in the
// last: 15 and 19 us, k = 32, d = 128 26 us, k = 1024, d = 128 38 us; now 13, 15, 20 and
// 27 us.
__global__ void __launch_bounds__(256) finalize_kernel(Accum acc, Centers c, StageState* st,
                                                       TrajDev tr, double* clus,
                                                       unsigned long long handle, int use_cond,
                                                       int stop)
{
    __shared__ FinalizeSmem sm;
    __shared__ int last;
    if (st->error) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            st->done = 1;
            if (use_cond) cudaGraphSetConditional(handle, 0u);
        }
        return;
    }
    const double inv = st->inv_scaleF;
    const int it = st->iter;
    for (int j = (int)(blockIdx.x + gridDim.x * (threadIdx.x >> 5)); j < c.k;
         j += (int)(gridDim.x * (blockDim.x >> 5)))
        finalize_center_warp(acc, c, inv, j, clus, tr, it);
    __syncthreads();
    for (int j = (int)(blockIdx.x + gridDim.x * threadIdx.x); j < c.k; j += (int)(gridDim.x * blockDim.x))
        finalize_divide(c.k, acc.cnt, inv, clus, j);
    if (gridDim.x > 1) {
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(&st->ticket, 1u) == gridDim.x - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
        if (threadIdx.x == 0) st->ticket = 0;
    } else {
        __syncthreads();
    }
    finalize_reduce_block(c.k, acc.cnt, st, tr, clus, sm);
    if (threadIdx.x == 0) {
        if (use_cond) cudaGraphSetConditional(handle, st->done ? 0u : 1u);
        if (stop && st->done) st->error = kErrStopped;
    }
}

// The stage's centers to a caller's device buffer, unless it failed.
__global__ void publish_centers_kernel(const StageState* st, const double* __restrict__ c64,
                                       long long count, double* __restrict__ out)
{
    if (st->error != 0 && st->error != kErrStopped) return;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < count;
         e += (long long)gridDim.x * blockDim.x)
        out[e] = c64[e];
}

constexpr int kRecheckThreads = 256;
constexpr int kRecheckCache = 1024;     // pass-1 values kept per warp (k <= 1024)

// Warps of the grid share the listed points (see recheck_warps), or blocks do when
// there are many centers and no more points than warps (recheck_point_block).
// More centers than kRecheckCache have two launches, of which one has work: kBlocks for
// the points that blocks take, kLarge for those of warps (in one kernel the block form
// is slower, n = 1e5, d = 100, k = 5000 3.2 -> 3.5 ms).  kBlocks keeps the code of kAll and
// leaves it by a flag: without that code it is given 40 registers, fewer loads in
// flight and 3.3 ms.
enum RecheckKind { kAll, kBlocks, kLarge };
constexpr int kOnlyBlocks = 2;          // in settles
template <RecheckKind KIND>
__global__ void __launch_bounds__(kRecheckThreads) recheck_kernel(const float* __restrict__ X, int d, Centers c,
                               int* __restrict__ labels, const int* __restrict__ list,
                               StageState* st, Accum acc, int settles)
{
    constexpr int W = kRecheckThreads / 32;
    __shared__ float cache[W * kRecheckCache];
    __shared__ RecheckBlockSmem sm;
    if (st->error) return;
    const long long nw = (long long)gridDim.x * W;
    if (c.k >= 256 && c.kpad <= W * kRecheckCache && st->recheck_count <= nw) {
        if constexpr (KIND != kLarge) {
            const int count = st->recheck_count;
            long long settled = 0;
            for (int p = blockIdx.x; p < count; p += gridDim.x)
                settled += recheck_point_block(X, d, c, labels, list[p], st, acc, cache, sm) ? 1 : 0;
            if ((KIND == kBlocks ? settles & 1 : settles) && settled && threadIdx.x == 0)
                atomicAdd(reinterpret_cast<unsigned long long*>(&st->rechecked_total),
                          (unsigned long long)(-settled));
        }
        return;
    }
    if (KIND == kBlocks && (settles & kOnlyBlocks)) return;
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    recheck_warps<KIND == kLarge>(X, d, c, labels, list, st, acc, gw, nw,
                                  cache + (threadIdx.x >> 5) * kRecheckCache, kRecheckCache, settles);
}

}  // namespace

static int grid_for(long long work, int threads, int sm_count, int per_sm)
{
    long long g = (work + threads - 1) / threads;
    long long cap = (long long)sm_count * per_sm;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

int launch_maxabs(const float* X, long long n, int d, StageState* st, cudaStream_t s,
                  int sm_count)
{
    const long long count = n * d;
    int vec4 = ((reinterpret_cast<uintptr_t>(X) & 15) == 0) ? 1 : 0;
    ++g_launches;
    maxabs_kernel<<<grid_for(count / 4 + 1, 256, sm_count, 8), 256, 0, s>>>(X, count, vec4, st);
    KM2_CUDA(cudaGetLastError());
    return KMEANS2_OK;
}

int launch_qsum(const float* X, long long n, int d, StageState* st, cudaStream_t s, int sm_count)
{
    const long long count = n * d;
    if (count <= 0) return KMEANS2_OK;
    int vec4 = ((reinterpret_cast<uintptr_t>(X) & 15) == 0) ? 1 : 0;
    ++g_launches;
    qsum_kernel<<<grid_for(count / 4 + 1, 256, sm_count, 8), 256, 0, s>>>(X, count, vec4, st);
    KM2_CUDA(cudaGetLastError());
    return KMEANS2_OK;
}

__global__ void recheck_reset_kernel(StageState* st)
{
    st->rechecked_total += st->recheck_count;
    st->listed_total += st->recheck_count;
    st->recheck_count = 0;
}

int launch_recheck_reset(StageState* st, cudaStream_t s)
{
    ++g_launches;
    recheck_reset_kernel<<<1, 1, 0, s>>>(st);
    KM2_CUDA(cudaGetLastError());
    return KMEANS2_OK;
}

int launch_gather(const float* X, int d, const long long* subset, long long m, float* Xs,
                  StageState* st, cudaStream_t s, int sm_count)
{
    ++g_launches;
    gather_kernel<<<grid_for(m * d, 256, sm_count, 8), 256, 0, s>>>(X, d, subset, m, Xs, st);
    KM2_CUDA(cudaGetLastError());
    return KMEANS2_OK;
}

int launch_init_centers(const float* Xs, int d, const long long* pos, int k, double* c64,
                        cudaStream_t s)
{
    long long total = (long long)k * d;
    int grid = (int)((total + 255) / 256);
    if (grid > 4096) grid = 4096;
    ++g_launches;
    init_centers_kernel<<<grid, 256, 0, s>>>(Xs, d, pos, k, c64);
    KM2_CUDA(cudaGetLastError());
    return KMEANS2_OK;
}

int launch_stage_begin(const Centers& c, const Accum& acc, StageState* st, double tol,
                       int max_iter, cudaStream_t s)
{
    const long long cn_len = center_norm_len(c.k, c.kpad);
    const long long work = std::max((long long)c.k * 32, (long long)c.dpad * c.kpad / 4);
    ++g_launches;
    stage_begin_kernel<<<(int)std::min(1024ll, (work + 255) / 256), 256, 0, s>>>(c, acc, st, tol,
                                                                               max_iter, cn_len);
    KM2_CUDA(cudaGetLastError());
    return KMEANS2_OK;
}

int launch_finalize(const Accum& acc, const Centers& c, StageState* st, const TrajDev& tr,
                    double* clus, unsigned long long cond_handle, int use_cond, int stop,
                    cudaStream_t s)
{
    ++g_launches;
    // one CTA for a handful of centers (no hand-over to a last CTA), else one
    // center per CTA up to about one CTA per SM
    finalize_kernel<<<c.k <= 8 ? 1 : std::min(c.k, 152), 256, 0, s>>>(acc, c, st, tr, clus,
                                                                     cond_handle, use_cond, stop);
    KM2_CUDA(cudaGetLastError());
    return KMEANS2_OK;
}

int launch_publish_centers(const StageState* st, const double* c64, long long count, double* out,
                           cudaStream_t s)
{
    ++g_launches;
    publish_centers_kernel<<<(int)std::min(152ll, (count + 255) / 256), 256, 0, s>>>(st, c64, count, out);
    KM2_CUDA(cudaGetLastError());
    return KMEANS2_OK;
}

int launch_recheck(const float* X, int d, const Centers& c, int* labels, const int* list,
                   StageState* st, const Accum& acc, int settles, cudaStream_t s, int sm_count)
{
    const int grid = sm_count * 4;
    if (c.kpad <= kRecheckCache) {
        ++g_launches;
        recheck_kernel<kAll><<<grid, kRecheckThreads, 0, s>>>(X, d, c, labels, list, st, acc, settles);
    } else {
        g_launches += 2;
        recheck_kernel<kBlocks><<<grid, kRecheckThreads, 0, s>>>(X, d, c, labels, list, st, acc,
                                                                settles | kOnlyBlocks);
        recheck_kernel<kLarge><<<grid, kRecheckThreads, 0, s>>>(X, d, c, labels, list, st, acc, settles);
    }
    KM2_CUDA(cudaGetLastError());
    return KMEANS2_OK;
}

}  // namespace km2
