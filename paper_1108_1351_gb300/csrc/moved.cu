// moved.cu -- the cluster sums of the 16-bit tensor-core forms.  Their k d words do
// not fit shared memory, and adding every moved row's coordinates to the global
// words (4 d 64-bit reductions per moved row) bound the distance kernel by the
// L2's reduction rate: n = 1e6, d = 128, k = 1024, FP16, first pass 2.47 ms.  The
// distance kernel therefore lists its moved rows and counts them by cluster
// (0.24 ms); one kernel here sorts the list (0.08 ms: a counting sort over 2 k
// bins: joined and left), the next adds each run of sorted rows in registers, with
// one set of reductions per run and cluster (0.24 ms).  The integer sums do not
// depend on the order.  Two launches, so that a pass that moves nothing pays
// little (5 us); a histogram and a scan kernel of their own cost 10 us more.
#include <algorithm>
#include <cstdint>

#include "api_internal.h"

namespace km2 {

namespace {

constexpr int kThreads = 256;
constexpr int kRun = 32;              // most sorted entries a warp adds up
constexpr int kMaxD = 128;

// Row and bin of every listed change, sorted by bin.  Each CTA scans the 2 k counts
// itself (8 KB at k = 1024) instead of waiting for a scan by one CTA.
__global__ void __launch_bounds__(kThreads) moved_scatter_kernel(MovedRows mv, const int* __restrict__ labels,
                                                                 int k, const StageState* st)
{
    __shared__ unsigned off[2 * kMovedMaxK];
    __shared__ unsigned ws[kThreads / 32];
    if (st->error) return;
    const unsigned count = min(mv.state[0], mv.cap);
    if (blockIdx.x * kThreads >= count) {
        if (blockIdx.x == 0 && threadIdx.x == 0) mv.state[1] = 0;
        return;
    }
    const int bins = 2 * k, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int b = threadIdx.x; b < bins; b += kThreads) off[b] = mv.hist[b];
    __syncthreads();
    const int per = (bins + kThreads - 1) / kThreads;
    const int b0 = min(bins, (int)threadIdx.x * per), b1 = min(bins, b0 + per);
    unsigned sum = 0;
    for (int b = b0; b < b1; ++b) sum += off[b];
    unsigned incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    unsigned pos = incl - sum;
    for (int w = 0; w < warp; ++w) pos += ws[w];
    for (int b = b0; b < b1; ++b) {
        const unsigned c = off[b];
        off[b] = pos;
        pos += c;
    }
    if (blockIdx.x == 0 && threadIdx.x == kThreads - 1) mv.state[1] = pos;
    __syncthreads();
    for (unsigned e = blockIdx.x * kThreads + threadIdx.x; e < count; e += gridDim.x * kThreads) {
        const int2 it = mv.moved[e];
        const int nl = labels[it.x], ol = it.y;
        mv.sorted[off[nl] + atomicAdd(mv.cur + nl, 1u)] = make_int2(it.x, nl);
        if (ol >= 0)
            mv.sorted[off[k + ol] + atomicAdd(mv.cur + k + ol, 1u)] = make_int2(it.x, k + ol);
    }
}

// A warp per run of sorted entries, lanes over coordinates (d <= 128); a short list
// is cut into shorter runs, so that the whole chip adds it.  Also the counts'
// change, and the histogram, cursors and list length back to zero (after an
// error as well: a shard's next pass starts from an empty list).
__global__ void __launch_bounds__(kThreads) moved_sum_kernel(const float* __restrict__ X, int d,
                                                             MovedRows mv, int k, Accum acc,
                                                             const StageState* st)
{
    constexpr int Q = kMaxD / 32;
    const bool ok = st->error == 0;
    const unsigned total = mv.state[1];
    for (int b = blockIdx.x * kThreads + threadIdx.x; b < 2 * k; b += gridDim.x * kThreads) {
        const unsigned c = mv.hist[b];
        if (c == 0) continue;
        mv.hist[b] = 0;
        mv.cur[b] = 0;
        if (ok) atomicAdd(acc.cnt + (b < k ? b : b - k), b < k ? (unsigned long long)c : 0ull - c);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) mv.state[0] = 0;
    if (!ok) return;
    const int lane = threadIdx.x & 31;
    const float scale = st->scaleF;
    const unsigned nw = gridDim.x * (kThreads / 32);
    const unsigned run = min((unsigned)kRun, max(1u, total / nw));
    for (unsigned e0 = (blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * run; e0 < total; e0 += nw * run) {
        const int cnt = (int)min(run, total - e0);
        const int2 it = lane < cnt ? mv.sorted[e0 + lane] : make_int2(0, 0);
        long long s[Q] = {};
        int bin = __shfl_sync(0xffffffffu, it.y, 0);
        auto flush = [&]() {
            const bool join = bin < k;
            const long long base = (long long)(join ? bin : bin - k) * d;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int t = lane + 32 * q;
                if (t < d && s[q]) split_add(acc.s_lo + base + t, acc.s_hi + base + t, join ? s[q] : -s[q]);
                s[q] = 0;
            }
        };
        for (int i = 0; i < cnt; i += 4) {           // four rows' loads in flight
            float v[4][Q];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = __shfl_sync(0xffffffffu, it.x, (i + u) & 31);
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const int t = lane + 32 * q;
                    v[u][q] = (t < d && i + u < cnt) ? __ldg(X + (long long)r * d + t) : 0.0f;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int b = __shfl_sync(0xffffffffu, it.y, (i + u) & 31);
                if (i + u < cnt && b != bin) {
                    flush();
                    bin = b;
                }
#pragma unroll
                for (int q = 0; q < Q; ++q) s[q] += to_fixed(v[u][q], scale);
            }
        }
        flush();
    }
}

}  // namespace

int launch_moved_sums(const float* X, long long n, int d, const MovedRows& mv, int k, const int* labels,
                      const StageState* st, const Accum& acc, cudaStream_t s, int sm_count)
{
    if (!mv.moved) return KMEANS2_OK;
    const int grid = (int)std::max(1ll, std::min((long long)sm_count * 4, (n + kThreads - 1) / kThreads));
    const int sums = (int)std::max(1ll, std::min((long long)sm_count * 6, (2 * n + 7) / 8));
    g_launches += 2;
    moved_scatter_kernel<<<grid, kThreads, 0, s>>>(mv, labels, k, st);
    moved_sum_kernel<<<sums, kThreads, 0, s>>>(X, d, mv, k, acc, st);
    KM2_CUDA(cudaGetLastError());
    return KMEANS2_OK;
}

}  // namespace km2
