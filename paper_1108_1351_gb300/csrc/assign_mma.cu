// assign_mma.cu -- the FP32 form's fused distance kernel with a tensor-core
// screen: split-FP16 products (22 significant bits per operand, FP32
// accumulation) on mma.sync decide every row whose best center is separated by
// more than their bound; the rest are decided by the FP32 FMA chain in the same
// warp, and what that leaves open by the FP64 recheck (mma_dev.cuh).  Labels,
// sums and J equal those of the CUDA-core kernels (assign_fp32.cu) bit for bit.
//
// assign_mma_ring (8 <= d <= 128): a warp takes 32 or 64 rows at a time from its own
// ring of cp.async stages in shared memory (rows as they lie in X, and the old
// labels); the centers' fragments stay in shared memory for the whole launch.
// Warps never wait for one another except to flush the partial sums.  Shapes
// whose centers do not fit beside the rings go to the CUDA-core kernels, and so do the
// later passes of a stage whose first ones leave too many rows open (review_screen):
// data far from the origin, whose bound grows with ||x||^2.
//
// What bounds it: instruction issue and register ports for d <= 16 (at d = 8, k =
// 32 it reads 3.1 TB/s), the legacy tensor rate (an MMA of 16 x 8 x 16 takes 8
// cycles per SM sub-partition) for wider rows, DRAM for few centers (d = 128, k =
// 32: 4.4 TB/s).  Per converged pass against the CUDA-core kernels (GB300; us):
//   n 2e7 d 8 k 32   325 -> 233      n 2e6 d 32 k 200   969 -> 237
//   n 1e7 d 12 k 16  216 -> 140      n 1e6 d 37 k 100   343 -> 115
//   n 4e6 d 8 k 256  428 -> 272      n 1e6 d 64 k 200   842 -> 210
//   n 4e6 d 16 k 100 378 -> 200      n 1e6 d 128 k 32   835 -> 119
//   n 1e6 d 16 k 1000 783 -> 360     n 5e5 d 128 k 100  423 -> 131
// Tried and dropped: 32 rows at a time at d = 8 (250); work handed out to warps
// dynamically (balance better, ~45 more instructions per 32 rows: 275); the
// candidate test as saturated FFMAs (250); the same screen on tcgen05 with one
// row per lane (d 8 k 32: 296, with warpgroup barriers and 330 instructions per
// 32 rows against 274; d 32 k 200: 321; d 64 k 200: 511); d < 8 (precision, see
// mma_dev.cuh).
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cstdint>

#include "api_internal.h"
#include "mma_dev.cuh"

namespace km2 {

namespace {

constexpr int kSmemCap = 224 * 1024;       // dynamic shared memory of an SM for these kernels

// Kernel shape by padded dimension.  d <= 16: 8 warps, 2 or 3 CTAs per SM, rings of
// 2 or 3 stages per warp.  Wider rows (WIDE): the A registers grow with d, so one
// CTA of as many warps as the registers hold; one stage per warp, refilled as soon
// as its rows are in registers (the MMAs of 32 rows take longer than the copy).
template <int DP, bool SINGLE>
struct RingCfg {
    static constexpr bool WIDE = DP > 16;
    static constexpr int W = DP <= 16 ? 8 : DP <= 32 ? 16 : DP <= 64 ? 12 : 8;   // warps
    static constexpr int THREADS = 32 * W;
    static constexpr int MINB = WIDE ? 1 : SINGLE ? 3 : 2;
    static constexpr int S = DP <= 8 ? 3 : DP <= 16 ? 2 : 1;                     // stages
};

__device__ __forceinline__ void cp_async16_zfill(unsigned sdst, const void* gsrc, int bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sdst), "l"(gsrc), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async16_u32(unsigned sdst, const void* gsrc)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sdst), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async4_u32(unsigned sdst, const void* gsrc)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sdst), "l"(gsrc) : "memory");
}

template <int N>
__device__ __forceinline__ void cp_async_wait_group()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// UNIT: rows a warp takes at a time (32 where n is too small to give every warp 64).
// DENSE (d <= 16): units with many open rows are decided a lane per row, and the open
// rows are counted.  A kernel of its own for a stage's first passes, whose count
// says whether the later ones keep the screen (review_screen): the code it adds
// costs the others 3 to 7 % (n = 1e8, d = 8, k = 32, a fit 65.6 -> 67.6 ms).
template <int DP, int NT, bool SINGLE, bool FULL, int UNIT, bool DENSE>
__global__ void __launch_bounds__((RingCfg<DP, SINGLE>::THREADS), (RingCfg<DP, SINGLE>::MINB))
assign_mma_ring(const float* __restrict__ X, long long n, Centers c, int* __restrict__ labels,
                StageState* st, Accum acc, int* __restrict__ list, int ntiles, int use_sacc)
{
    using R = RingCfg<DP, SINGLE>;
    constexpr int S = R::S, kWarps = R::W, kThreads = R::THREADS;
    constexpr bool WIDE = R::WIDE;
    constexpr int H = UNIT / 32;
    static_assert(!WIDE || UNIT == 32, "wide rows: one 32-row block per warp and step");
    static_assert(!(WIDE && DENSE), "wide rows: the recheck decides the open ones");
    constexpr int kFlushSteps = kFlushPoints / (kWarps * UNIT);   // steps per int64 partial
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_open;                               // DENSE: rows the screen left open
    if (st->error) return;
    const int k = c.k, d = FULL ? DP : c.d;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const unsigned stage_bytes = 4 * UNIT * (d + 1);       // rows, then labels
    uint32_t* sb = reinterpret_cast<uint32_t*>(smem);
    float* sn = reinterpret_cast<float*>(sb + (size_t)ntiles * MmaCfg<DP>::BW * 32);
    unsigned char* ring = reinterpret_cast<unsigned char*>(sn + ntiles * 8) +
                          (size_t)warp * S * stage_bytes;
    long long* sacc = reinterpret_cast<long long*>(reinterpret_cast<unsigned char*>(sn + ntiles * 8) +
                                                   (size_t)kWarps * S * stage_bytes);
    int* scnt = reinterpret_cast<int*>(sacc + (size_t)k * d);
    const bool delta = st->mode == kModeDelta;
    const float scaleF = st->scaleF;
    const float thr_base = 2.0f * st->cmax2;
    const MmaScale ms = mma_scale(st, d, MmaCfg<DP>::KS);

    // step i of this CTA: rows [T tile_rows, + tile_rows), T = blockIdx.x + i gridDim.x;
    // the warp's unit starts UNIT * warp rows into it (n < 2^31)
    constexpr int tile_rows = kWarps * UNIT;
    const int steps = (int)((n + tile_rows - 1) / tile_rows);
    constexpr int NQ = (UNIT * DP + 127) / 128;         // 16-byte copies per lane and stage, at most
    const long long row_first = (long long)blockIdx.x * tile_rows + warp * UNIT;
    const unsigned char* xsrc = reinterpret_cast<const unsigned char*>(X + row_first * d) + 16 * lane;
    const int* lsrc = labels + row_first + lane;
    const long long rstep = (long long)gridDim.x * tile_rows;
    long long left_issue = n - row_first;                // rows from the next issue's first one on
    const unsigned ring_u32 = smem_u32(ring);
    // the next unit's rows and labels (in a full pass those are read and not
    // used) -> the stage at byte offset `so` of the ring; rows past n are
    // zero-filled
    auto issue = [&](unsigned so) {
        const unsigned dst = ring_u32 + so + 16 * lane, ldst = ring_u32 + so + 4 * UNIT * d + 4 * lane;
        if (left_issue >= UNIT) {
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (lane + 32 * q < UNIT / 4 * d) cp_async16_u32(dst + 512 * q, xsrc + 512 * q);
            cp_async4_u32(ldst, lsrc);
            if (H == 2) cp_async4_u32(ldst + 128, lsrc + 32);
        } else {
            const int rows = (int)max(0ll, min(left_issue, (long long)UNIT));
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int have = min(16, max(0, rows * d * 4 - 16 * (lane + 32 * q)));
                if (lane + 32 * q < UNIT / 4 * d)
                    cp_async16_zfill(dst + 512 * q, have ? xsrc + 512 * q : reinterpret_cast<const unsigned char*>(X), have);
            }
            if (lane < rows) cp_async4_u32(ldst, lsrc);
            if (H == 2 && lane + 32 < rows) cp_async4_u32(ldst + 128, lsrc + 32);
        }
        cp_async_commit();
        xsrc += rstep * d * 4;
        lsrc += rstep;
        left_issue -= rstep;
    };
    // WIDE: the first unit now, each next one once the stage's rows are in registers
#pragma unroll
    for (int s = 0; s < (WIDE ? 1 : S - 1); ++s) issue(s * stage_bytes);

    if (DENSE && tid == 0) s_open = 0;
    mma_load_centers<DP>(c, ntiles, ms, sb, sn);
    if (use_sacc) {
        for (int e = tid; e < k * d; e += kThreads) sacc[e] = 0;
        for (int e = tid; e < k; e += kThreads) scnt[e] = 0;
    }
    __syncthreads();

    unsigned so = 0;                                     // the current stage's offset
    const unsigned ring_bytes = S * stage_bytes;
    int to_flush = kFlushSteps;
    for (int step = blockIdx.x; step < steps; step += gridDim.x) {
        if (!WIDE) issue(so == 0 ? ring_bytes - stage_bytes : so - stage_bytes);
        cp_async_wait_group<S - 1>();
        __syncwarp();
        const float* xr = reinterpret_cast<const float*>(ring + so);
        const int* lr = reinterpret_cast<const int*>(ring + so + 4 * UNIT * d);
        const long long row0 = (long long)step * tile_rows + warp * UNIT;
        const int rows = (int)min((long long)UNIT, n - row0);   // may be <= 0 in the last step

        // row of this lane in half h: 32 h + 8 t + g
        int lab[2], old[2];
        bool open[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h >= H) { lab[h] = old[h] = -1; open[h] = false; continue; }
            uint32_t A[2][MmaCfg<DP>::AREG];
            float xmax = 0.0f;
            mma_load_rows<DP, FULL>(xr + 32 * h * d, d, g, t, 0, ms.sx, A[0], xmax);
            mma_load_rows<DP, FULL>(xr + 32 * h * d, d, g, t, 1, ms.sx, A[1], xmax);
            old[h] = delta ? lr[32 * h + 8 * t + g] : -1;
            if (WIDE && delta) {
                __syncwarp();            // every lane has read the stage
                issue(0);
            }
            lab[h] = mma_decide<DP, NT, SINGLE>(A, sb, sn, ntiles, lane, mma_thr(ms, xmax), open[h]);
            if (32 * h + 8 * t + g >= rows) { open[h] = false; lab[h] = old[h]; }
        }
        if (WIDE) {
            // the recheck kernel decides the open rows: its FP32 pass over k d center
            // values finds them in L1, which shared memory leaves little of here
            recheck_append(open[0], (int)(row0 + 8 * t + g), list, &st->recheck_count);
            if (open[0]) lab[0] = old[0];
        } else if (__any_sync(0xffffffffu, open[0] || open[1])) {
#pragma unroll
            for (int h = 0; h < H; ++h) {
                unsigned todo = __ballot_sync(0xffffffffu, open[h]);
                bool listed = false;
                if constexpr (DENSE) {
                    if (lane == 0) atomicAdd(&s_open, __popc(todo));
                    if (__popc(todo) >= lanes_from(d, k)) {
                        const int l = decide_fp32_lanes<DP, FULL>(xr + (32 * h + 8 * t + g) * d, d, c.cnorm, c.c32t,
                                                                  c.kpad, k, thr_base);
                        if (open[h]) { lab[h] = l; listed = l < 0; }
                        todo = 0;
                    }
                }
#pragma unroll 1
                while (todo) {
                    const int o = __ffs(todo) - 1;
                    todo &= todo - 1;
                    bool op;
                    const int l = decide_fp32_row(X + (row0 + 32 * h + 8 * (o & 3) + (o >> 2)) * d, d, c,
                                                  thr_base, op);
                    if (lane == o) { lab[h] = l; listed = op; }
                }
                recheck_append(listed, (int)(row0 + 32 * h + 8 * t + g), list, &st->recheck_count);
                if (listed) lab[h] = old[h];             // the recheck moves it
            }
        }
        if (__any_sync(0xffffffffu, lab[0] != old[0] || lab[1] != old[1])) {
            auto add = [&](int lo, int ol, int dim, float xv) {
                const long long v = to_fixed(xv, scaleF);
                if (use_sacc) {
                    atomicAdd(reinterpret_cast<unsigned long long*>(sacc + lo * d + dim), (unsigned long long)v);
                    if (ol >= 0)
                        atomicAdd(reinterpret_cast<unsigned long long*>(sacc + ol * d + dim), (unsigned long long)(-v));
                } else {
                    split_add(acc.s_lo + (long long)lo * d + dim, acc.s_hi + (long long)lo * d + dim, v);
                    if (ol >= 0)
                        split_add(acc.s_lo + (long long)ol * d + dim, acc.s_hi + (long long)ol * d + dim, -v);
                }
            };
            auto count = [&](int lo, int ol) {
                if (use_sacc) {
                    atomicAdd(scnt + lo, 1);
                    if (ol >= 0) atomicAdd(scnt + ol, -1);
                } else {
                    atomicAdd(acc.cnt + lo, 1ull);
                    if (ol >= 0) atomicAdd(acc.cnt + ol, ~0ull);
                }
            };
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const bool moved = lab[h] != old[h] && label_ok(lab[h], k, st) && old_label_ok(old[h], k, st);
                unsigned mv = __ballot_sync(0xffffffffu, moved);
                if (moved) {
                    labels[row0 + 32 * h + 8 * t + g] = lab[h];
                    count(lab[h], old[h]);
                }
                // 32 / LPR moved rows at a time, LPR lanes per row, a coordinate each: at most
                // 32 / LPR lanes meet on one word (a lane per row is slower in full
                // passes: 8.2 against 3.8 ms for n = 1e8, d = 8, k = 32, where a few large
                // clusters take most rows)
                constexpr int LPR = DP < 32 ? DP : 32;
#pragma unroll 1
                while (mv) {
                    int o = -1;
#pragma unroll
                    for (int q = 0; q < 32 / LPR; ++q) {
                        if (lane / LPR == q) o = __ffs(mv) - 1;
                        mv &= mv - 1;              // 0 stays 0
                    }
                    const int src = o < 0 ? 0 : o;
                    const int lo = __shfl_sync(0xffffffffu, lab[h], src);
                    const int ol = __shfl_sync(0xffffffffu, old[h], src);
                    if (o >= 0) {
                        const int r = 32 * h + 8 * (o & 3) + (o >> 2);
                        if (WIDE) {                // delta: the stage holds other rows by now
                            const float* xg = delta ? X + (row0 + r) * d : xr + r * d;
                            for (int dim = lane; dim < d; dim += 32) add(lo, ol, dim, xg[dim]);
                        } else if (lane % LPR < d) {
                            add(lo, ol, lane % LPR, xr[r * d + lane % LPR]);
                        }
                    }
                    __syncwarp();
                }
            }
        }
        __syncwarp();   // every lane is done with the stage before it is refilled
        if (WIDE && !delta) issue(0);   // a full pass adds every row's coordinates from the stage
        so = so + stage_bytes == ring_bytes ? 0 : so + stage_bytes;

        // static flush schedule: at most 2^16 rows per int64 partial
        if (use_sacc && (--to_flush == 0 || step + (int)gridDim.x >= steps)) {
            to_flush = kFlushSteps;
            __syncthreads();
            for (int e = tid; e < k * d; e += kThreads) {
                const long long v = sacc[e];
                if (v) {
                    split_add(acc.s_lo + e, acc.s_hi + e, v);
                    sacc[e] = 0;
                }
            }
            for (int e = tid; e < k; e += kThreads) {
                const int v = scnt[e];
                if (v) {
                    atomicAdd(acc.cnt + e, (unsigned long long)(long long)v);
                    scnt[e] = 0;
                }
            }
            __syncthreads();
        }
    }
    cp_async_wait_group<0>();
    if constexpr (DENSE) {
        __syncthreads();
        if (tid == 0 && s_open) atomicAdd(&st->open_rows, (unsigned long long)s_open);
    }
}

template <int DP, bool SINGLE, int UNIT>
size_t ring_bytes(int d) { return (size_t)RingCfg<DP, SINGLE>::W * RingCfg<DP, SINGLE>::S * 4 * UNIT * (d + 1); }

template <int DP, int NT, bool SINGLE, bool FULL, int UNIT, bool DENSE>
int launch_ring_u(const float* X, long long n, const Centers& c, int* labels, StageState* st,
                  const Accum& acc, int* list, int ntiles, cudaStream_t s, int sm_count)
{
    using R = RingCfg<DP, SINGLE>;
    const size_t base = mma_center_bytes(DP, ntiles) + ring_bytes<DP, SINGLE, UNIT>(c.d);
    const size_t sums = (size_t)c.k * c.d * 8 + (size_t)c.k * 4;
    const int use_sacc = base + sums <= (size_t)kSmemCap;
    const size_t sm = base + (use_sacc ? sums : 0);
    const void* kfn = (const void*)assign_mma_ring<DP, NT, SINGLE, FULL, UNIT, DENSE>;
    KM2_TRY(set_max_dynamic_smem(kfn, kSmemCap));
    int per_sm = 0;
    KM2_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, R::THREADS, sm));
    if (per_sm < 1) return KMEANS2_ERR_UNSUPPORTED;
    const long long steps = (n + R::W * UNIT - 1) / (R::W * UNIT);
    const int grid = (int)std::max(1ll, std::min((long long)sm_count * per_sm, steps));
    ++g_launches;
    assign_mma_ring<DP, NT, SINGLE, FULL, UNIT, DENSE><<<grid, R::THREADS, sm, s>>>(X, n, c, labels, st, acc,
                                                                           list, ntiles, use_sacc);
    KM2_CUDA(cudaGetLastError());
    return KMEANS2_OK;
}

template <int DP, int NT, bool SINGLE>
int launch_ring(const float* X, long long n, const Centers& c, int* labels, StageState* st,
                const Accum& acc, int* list, int ntiles, int first, cudaStream_t s, int sm_count)
{
    // 64 rows per warp and step once every warp of two or three CTAs per SM gets
    // some; below, 32 (too few warps otherwise)
    const bool small = n < (long long)sm_count * RingCfg<DP, SINGLE>::MINB * RingCfg<DP, SINGLE>::W * 64;
#define KM2_RING(FULL_, UNIT_, DENSE_) \
    return launch_ring_u<DP, NT, SINGLE, FULL_, UNIT_, DENSE_>(X, n, c, labels, st, acc, list, ntiles, s, sm_count)
#define KM2_RING_NARROW(FULL_)                 \
    if (small && first) KM2_RING(FULL_, 32, true); \
    if (small) KM2_RING(FULL_, 32, false);     \
    if (first) KM2_RING(FULL_, 64, true);      \
    KM2_RING(FULL_, 64, false)
    if constexpr (DP > 16) KM2_RING(false, 32, false);
    if constexpr (DP <= 16) if (c.d == DP) { KM2_RING_NARROW(true); }
    if constexpr (DP == 16) { KM2_RING_NARROW(false); }
#undef KM2_RING_NARROW
#undef KM2_RING
    return KMEANS2_ERR_UNSUPPORTED;
}

template <int DP>
int launch_ring_k(const float* X, long long n, const Centers& c, int* labels, StageState* st,
                  const Accum& acc, int* list, int first, cudaStream_t s, int sm_count)
{
    if constexpr (DP > 64) {
        // two accumulators per block (mma_chunk): chunks of 16 centers
        if (c.k <= 16) return launch_ring<DP, 2, true>(X, n, c, labels, st, acc, list, 2, first, s, sm_count);
        return launch_ring<DP, 2, false>(X, n, c, labels, st, acc, list, (c.k + 15) / 16 * 2, first, s, sm_count);
    } else {
        if constexpr (DP <= 16)
            if (c.k <= 16) return launch_ring<DP, 2, true>(X, n, c, labels, st, acc, list, 2, first, s, sm_count);
        if (c.k <= 32) return launch_ring<DP, 4, true>(X, n, c, labels, st, acc, list, 4, first, s, sm_count);
        return launch_ring<DP, 4, false>(X, n, c, labels, st, acc, list, (c.k + 31) / 32 * 4, first, s, sm_count);
    }
}

#define KM2_RING_DPS(X) X(8) X(16) X(32) X(48) X(64) X(96) X(128)

}  // namespace

// d from 8 on: see the precision figures in mma_dev.cuh.
int assign_mma_supported(int d, int k, const float* X)
{
    if ((reinterpret_cast<uintptr_t>(X) & 15) != 0 || d < 8 || d > 128) return 0;
    switch (mma_dp(d)) {
#define KM2_CASE(DD) case DD: return mma_center_bytes(DD, (k + 31) / 32 * 4) + \
        ring_bytes<DD, false, (DD > 16 ? 32 : 64)>(d) <= (size_t)kSmemCap;
        KM2_RING_DPS(KM2_CASE)
#undef KM2_CASE
        default: return 0;
    }
}

int launch_assign_mma(const float* X, long long n, int d, const Centers& c, int* labels,
                      StageState* st, const Accum& acc, int* list, int first, cudaStream_t s,
                      int sm_count)
{
    switch (mma_dp(d)) {
#define KM2_CASE(DD) case DD: return launch_ring_k<DD>(X, n, c, labels, st, acc, list, first, s, sm_count);
        KM2_RING_DPS(KM2_CASE)
#undef KM2_CASE
        default: return KMEANS2_ERR_UNSUPPORTED;
    }
}

}  // namespace km2
