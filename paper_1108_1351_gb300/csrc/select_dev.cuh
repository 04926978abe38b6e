// select_dev.cuh -- the Algorithm's random draws by one CTA: exact selection of the
// smallest SplitMix64 keys (sample.cu for the definition), for the jobs of a
// batch and for single fits small enough that the multi-kernel selection is all
// launches and one-CTA steps.
#pragma once

#include "common.cuh"

namespace km2 {

constexpr int kSampleThreads = 1024;

// Block-level exact radix select: ascending positions (relative to `off`) of
// the `want` smallest keys splitmix64_at(seed, off + i), i in [0, count).
static __device__ void select_block(unsigned long long seed, unsigned long long off, long long count,
                             long long want, long long* out)
{
    __shared__ unsigned int hist[256];
    __shared__ unsigned long long prefix;
    __shared__ long long need;
    __shared__ long long scan[kSampleThreads];
    if (threadIdx.x == 0) { prefix = 0; need = want; }
    __syncthreads();
    for (int pass = 0; pass < 8; ++pass) {
        const int shift = 56 - 8 * pass;
        for (int b = threadIdx.x; b < 256; b += blockDim.x) hist[b] = 0;
        __syncthreads();
        const unsigned long long pf = prefix;
        for (long long i = threadIdx.x; i < count; i += blockDim.x) {
            const unsigned long long key = splitmix64_at(seed, off + (unsigned long long)i);
            const bool match = pass == 0 || (key >> (shift + 8)) == (pf >> (shift + 8));
            if (match) atomicAdd(&hist[(key >> shift) & 255ull], 1u);
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            // eight bins per lane: the lane whose range holds the need-th key
            const long long nd = need;
            const int lane = threadIdx.x;
            long long sum = 0;
            for (int b = 0; b < 8; ++b) sum += hist[8 * lane + b];
            long long incl = sum;
            for (int o = 1; o < 32; o <<= 1) {
                const long long v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            long long acc = incl - sum;
            if (nd > acc && nd <= incl) {
                int b = 8 * lane;
                while (nd > acc + (long long)hist[b]) acc += hist[b++];
                prefix = pf | ((unsigned long long)b << shift);
                need = nd - acc;
            }
        }
        __syncthreads();
    }
    const unsigned long long T = prefix;     // the want-th smallest key (keys are distinct)
    const long long per = (count + blockDim.x - 1) / blockDim.x;
    const long long i0 = min(count, (long long)threadIdx.x * per), i1 = min(count, i0 + per);
    long long c = 0;
    for (long long i = i0; i < i1; ++i) c += splitmix64_at(seed, off + (unsigned long long)i) <= T;
    scan[threadIdx.x] = c;
    __syncthreads();
    if (threadIdx.x < 32) {
        // exclusive scan, 32 threads' counts per lane
        long long sum = 0;
        for (int t = 0; t < kSampleThreads / 32; ++t) sum += scan[threadIdx.x * (kSampleThreads / 32) + t];
        long long a = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const long long v = __shfl_up_sync(0xffffffffu, a, o);
            if ((int)threadIdx.x >= o) a += v;
        }
        a -= sum;
        for (int t = 0; t < kSampleThreads / 32; ++t) {
            const int e = threadIdx.x * (kSampleThreads / 32) + t;
            const long long v = scan[e];
            scan[e] = a;
            a += v;
        }
    }
    __syncthreads();
    long long o = scan[threadIdx.x];
    for (long long i = i0; i < i1; ++i)
        if (splitmix64_at(seed, off + (unsigned long long)i) <= T) out[o++] = i;
    __syncthreads();
}

// Ranks one CTA forms itself, k / 1024 times k keys per thread; more are left to
// a grid (k = 5000, n = 9,000, a fit: 5.7 ms with the ranks by one CTA, 2.1 by a grid).
constexpr int kRankOneCta = 256;

// Both draws: S_s (m ascending positions of [0, n)) and the initial centers (k
// positions of [0, m) in increasing key order); tmp: k positions of scratch, the
// centers' positions in ascending order (all there is for k > kRankOneCta).
static __device__ void sample_block(unsigned long long seed, long long n, long long m, int k,
                                    long long* subset, long long* pos, long long* tmp)
{
    select_block(seed, 0ull, n, m, subset);
    select_block(seed, (unsigned long long)n, m, k, tmp);
    if (k > kRankOneCta) return;
    for (int a = threadIdx.x; a < k; a += blockDim.x) {
        const unsigned long long ka = splitmix64_at(seed, (unsigned long long)(n + tmp[a]));
        int rank = 0;
        for (int b = 0; b < k; ++b)
            rank += splitmix64_at(seed, (unsigned long long)(n + tmp[b])) < ka;
        pos[rank] = tmp[a];
    }
}

}  // namespace km2
