// stage_dev.cuh -- block- and warp-level bodies of the per-stage steps, shared
// by the single-fit kernels (prep.cu) and the batched kernels (batched.cu) so
// that both run exactly the same arithmetic:
//   center_prep_block  FP32 / transposed copies of the FP64 centers, ||c||^2
//   stage_init_dev     fixed-point scales and loop state of one stage
//   finalize_*         new centers = cluster means (Lloyd's method, Section 4.1),
//                      largest movement (stop test, Sections 5-6), J (Eq. 3)
//   recheck_warps      FP64 re-evaluation of near-tie points (ties -> lowest index)
#pragma once

#include <cfloat>
#include <climits>

#include "common.cuh"

namespace km2 {

__device__ __forceinline__ double warp_sum_f64(double v)
{
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// FP32 copies and ||c_j||^2 of every center; st->cmax2 = max_j ||c_j||^2 rounded
// up.  Whole block; warps stride over centers.
// red: blockDim.x doubles of shared memory.
static __device__ void center_prep_block(Centers c, StageState* st, double* red)
{
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    double mx = 0.0;
    for (int j = warp; j < c.k; j += nw) {
        double nn = 0.0;
        for (int t = lane; t < c.d; t += 32) {
            double v = c.c64[(long long)j * c.d + t];
            nn = fma(v, v, nn);
            c.c32[(long long)j * c.d + t] = (float)v;
            c.c32t[(long long)t * c.kpad + j] = (float)v;
        }
        nn = warp_sum_f64(nn);
        if (lane == 0) c.cnorm[j] = (float)nn;
        mx = fmax(mx, nn);
    }
    red[threadIdx.x] = mx;
    __syncthreads();
    for (int s = blockDim.x >> 1; s; s >>= 1) {
        if ((int)threadIdx.x < s) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) st->cmax2 = __double2float_ru(red[0]);
    __syncthreads();
}

// One thread.  Loop state of a new stage and its fixed-point scales from
// st->maxabs_bits (max |x| of the stage's points).
static __device__ void stage_init_dev(StageState* st, int d, double tol, int max_iter)
{
    unsigned int b = st->maxabs_bits;
    st->mode = kModeFull;
    st->iter = 0;
    st->done = 0;
    st->converged = 0;
    st->max_iter = max_iter;
    st->tol = tol;
    st->recheck_count = 0;
    st->rechecked_total = 0;
    st->listed_total = 0;
    st->undecided16_total = 0;
    for (int w = 0; w < 4; ++w) st->q[w] = 0ull;
    st->J = 0.0;
    st->shift = 0.0;
    st->empty = 0;
    st->error = 0;
    if (b >= 0x7f800000u) {
        st->error = kErrNonFinite;
        st->done = 1;
        return;
    }
    float mx = __uint_as_float(b);
    int E = -126;
    if (mx > 0.0f) frexpf(mx, &E);          // mx < 2^E
    if (E > 50) {
        st->error = kErrRange;
        st->done = 1;
        return;
    }
    (void)d;
    int F = min(120, max(-100, 46 - E));
    st->F = F;
    st->scaleF = ldexpf(1.0f, F);
    st->inv_scaleF = ldexp(1.0, -F);
}

// ---------------------------------------------------------------- exact J
// Error-free transformations (Knuth's TwoSum, Dekker's FastTwoSum, and the
// FMA two-product) for the center-displacement term of J.
__device__ __forceinline__ void two_sum(double a, double b, double& s, double& e)
{
    s = a + b;
    const double bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ void fast_two_sum(double a, double b, double& s, double& e)
{
    s = a + b;
    e = b - (s - a);
}

// N c - s 2^-F for a center coordinate c (FP64), a cluster size N and the
// exact integer sum s of the cluster's fixed-point coordinates: N times the
// center's displacement from the cluster mean.  c N is split exactly into the
// double-word p + e (FMA two-product) and s 2^-F exactly into a1 + a2 (the
// 32-bit halves of s, scaled by powers of two), renormalised by TwoSum into
// the double-word b1 + b2; the two double-words are then added with the
// accurate double-word sum (two TwoSums, two renormalisations), whose relative
// error is below 3 * 2^-106 of the result however close c is to the mean.
__device__ __forceinline__ double displacement(double c, double N, __int128 s, double inv)
{
    const __int128 sh = s >> 32;                       // |sh| < 2^50: exact in FP64
    const double a1 = (double)(long long)sh * (inv * 4294967296.0);
    const double a2 = (double)(unsigned long long)(s - (sh << 32)) * inv;
    double b1, b2;
    two_sum(a1, a2, b1, b2);
    const double p = c * N;
    const double e = fma(c, N, -p);
    double s1, s2, t1, t2;
    two_sum(p, -b1, s1, s2);
    two_sum(e, -b2, t1, t2);
    s2 += t1;
    fast_two_sum(s1, s2, s1, s2);
    s2 += t2;
    fast_two_sum(s1, s2, s1, s2);
    return s1;
}

// 256-bit two's complement integers for the integer part of J.
struct U256 {
    unsigned long long w[4];
};

// a += v * 2^(64 limb), carries propagated to the top limb.
__device__ __forceinline__ void u256_add_at(U256& a, unsigned __int128 v, int limb)
{
    unsigned long long carry = 0;
    for (int i = limb; i < 4; ++i) {
        const unsigned long long add = (i == limb) ? (unsigned long long)v
                                     : (i == limb + 1) ? (unsigned long long)(v >> 64) : 0ull;
        const unsigned __int128 t = (unsigned __int128)a.w[i] + add + carry;
        a.w[i] = (unsigned long long)t;
        carry = (unsigned long long)(t >> 64);
    }
}

__device__ __forceinline__ void u256_neg(U256& a)
{
    unsigned long long carry = 1;
    for (int i = 0; i < 4; ++i) {
        const unsigned __int128 t = (unsigned __int128)(~a.w[i]) + carry;
        a.w[i] = (unsigned long long)t;
        carry = (unsigned long long)(t >> 64);
    }
}

// The signed value of a, rounded to FP64 (the top 128 significant bits are
// converted in one rounding; the rest is below 2^-64 of it).
__device__ __forceinline__ double u256_to_double(U256 a)
{
    const bool neg = (long long)a.w[3] < 0;
    if (neg) u256_neg(a);
    int top = 3;
    while (top > 0 && a.w[top] == 0) --top;
    double r;
    if (top == 0) {
        r = (double)a.w[0];
    } else {
        const unsigned __int128 hi = ((unsigned __int128)a.w[top] << 64) | a.w[top - 1];
        r = ldexp((double)hi, 64 * (top - 1));
        if (top >= 2) r += ldexp((double)a.w[top - 2], 64 * (top - 2));
    }
    return neg ? -r : r;
}

// One warp: the new center j (its cluster mean; an empty cluster keeps its
// center) with its FP32 copies and ||c_j||^2, and center j's terms of the
// movement and of J in clus (kClusSlots k words):
//   clus[j]          ||c_j' - c_j||^2
//   clus[k + j]      sum_t (N_j c_jt - s_jt 2^-F)^2 = N_j^2 ||c_j - mu_j||^2
//   clus[2k + j]     ||c_j'||^2
//   clus[3k + 3j..]  T_j as three 64-bit limbs
// where s_jt = the exact integer sum of the cluster's fixed-point coordinates,
// mu_j = s_j 2^-F / N_j its mean and T_j = ||s_j||^2; finalize_reduce_block divides.
// Iteration it's records of center j go to tr.centers / tr.counts when those are set.
static __device__ __forceinline__ void finalize_center_warp(const Accum& acc, const Centers& c,
                                                            double inv, int j, double* clus,
                                                            const TrajDev& tr, int it)
{
    const int k = c.k, d = c.d;
    const int lane = threadIdx.x & 31;
    const long long N = (long long)acc.cnt[j];
    const double Nd = (double)N;
    double diff2 = 0.0, dev2 = 0.0, nn = 0.0;
    // T_j = t_hi 2^64 + t_lo, partial per lane (no carries needed: t_lo gains
    // < 2^65 per coordinate, t_hi < 2^101)
    unsigned __int128 t_lo = 0, t_hi = 0;
    for (int t = lane; t < d; t += 32) {
        long long e = (long long)j * d + t;
        const unsigned long long lo = acc.s_lo[e], hi = acc.s_hi[e];
        const __int128 v = (__int128)(long long)hi * (__int128)4294967296LL + (__int128)lo;
        // v to FP64 in one rounding: |v >> 32| < 2^50, both halves exact
        const double S = fma((double)(long long)(v >> 32), 4294967296.0, (double)(unsigned)v) * inv;
        // carry the low word's upper half into the high word (same value):
        // every pass adds at most 2 n < 2^32 low parts below 2^32 each, so
        // the low word cannot wrap however many delta passes follow
        acc.s_lo[e] = lo & 0xffffffffull;
        acc.s_hi[e] = hi + (lo >> 32);
        double cv = c.c64[e];
        double cn = N > 0 ? S / Nd : cv;
        double df = cn - cv;
        diff2 = fma(df, df, diff2);
        nn = fma(cn, cn, nn);
        if (N > 0) {
            const unsigned __int128 a = (unsigned __int128)(v < 0 ? -v : v);   // < 2^82
            const unsigned long long al = (unsigned long long)a & 0xffffffffull;
            const unsigned __int128 ah = a >> 32;
            const unsigned __int128 m = 2 * ah * al;
            t_hi += ah * ah + (m >> 32);
            t_lo += ((m & 0xffffffffull) << 32) + (unsigned __int128)al * al;
            const double r = displacement(cv, Nd, v, inv);
            dev2 = fma(r, r, dev2);
        }
        c.c64[e] = cn;
        c.c32[e] = (float)cn;
        c.c32t[(long long)t * c.kpad + j] = (float)cn;
        if (tr.centers) tr.centers[(long long)it * k * d + e] = cn;
    }
    diff2 = warp_sum_f64(diff2);
    dev2 = warp_sum_f64(dev2);
    nn = warp_sum_f64(nn);
    t_lo = warp_sum_u128(t_lo);
    t_hi = warp_sum_u128(t_hi);
    if (lane == 0) {
        t_hi += t_lo >> 64;
        unsigned long long* qw = reinterpret_cast<unsigned long long*>(clus + 3 * k) + 3ll * j;
        qw[0] = (unsigned long long)t_lo;
        qw[1] = (unsigned long long)t_hi;
        qw[2] = (unsigned long long)(t_hi >> 64);
        clus[j] = diff2;
        clus[k + j] = dev2;
        clus[2 * k + j] = nn;
        c.cnorm[j] = (float)nn;
        if (tr.counts) tr.counts[(long long)it * k + j] = N;
    }
}

// floor(T / N) of a 192-bit T (three limbs, in place) for 0 < N < 2^32, and T mod
// N: long division by 32-bit digits, each quotient digit from an FP64 product
// with 1 / N (off by at most one: the digit is below 2^32 and the product's
// relative error below 2^-51) and corrected exactly.
__device__ __forceinline__ unsigned long long div192(unsigned long long (&T)[3], unsigned long long N)
{
    const double inv = 1.0 / (double)N;
    unsigned long long rem = 0, Q[3] = {0ull, 0ull, 0ull};
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        const unsigned long long digit = (T[i >> 1] >> (32 * (i & 1))) & 0xffffffffull;
        const unsigned long long x = (rem << 32) | digit;          // < N 2^32
        unsigned long long q = 0;
        if (x >= N) {
            q = (unsigned long long)((double)x * inv);
            long long r = (long long)(x - q * N);
            if (r < 0) { --q; r += (long long)N; }
            if (r >= (long long)N) { ++q; r -= (long long)N; }
            rem = (unsigned long long)r;
        } else {
            rem = x;
        }
        Q[i >> 1] |= q << (32 * (i & 1));
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) T[i] = Q[i];
    return rem;
}

// One thread: center j's division.  T_j becomes floor(T_j / N_j) in place, and
// clus[k + j] its remaining term of J, N_j ||c_j - mu_j||^2 - frac(T_j / N_j) 2^-2F
// (zeros for an empty cluster).
static __device__ __forceinline__ void finalize_divide(int k, const unsigned long long* cnt,
                                                       double inv, double* clus, int j)
{
    unsigned long long* qw = reinterpret_cast<unsigned long long*>(clus + 3 * k) + 3ll * j;
    const unsigned long long N = cnt[j];
    double term = 0.0;
    if ((long long)N > 0) {
        unsigned long long T[3] = {qw[0], qw[1], qw[2]};
        const unsigned long long rem = div192(T, N);
        const double Nd = (double)N;
        term = clus[k + j] / Nd - ((double)rem / Nd) * (inv * inv);
        qw[0] = T[0];
        qw[1] = T[1];
        qw[2] = T[2];
    }
    clus[k + j] = term;
}

struct FinalizeSmem {
    double r_shift[32];
    double r_J[256];
    double r_nn[32];
    int r_empty[32];
    unsigned __int128 r_q[32][3];
};

// Whole block of 256 threads, after every center's finalize_center_warp and
// finalize_divide: movement, J and loop control from clus (thread 0 updates st).
// J's floating terms are added in one fixed order, the one of a tree over 1024
// threads that stride over the centers.  The integer part of J, sum s^2 - sum_j
// floor(T_j / N_j), is exact (256-bit); it is rounded to FP64 once and added to the
// sum of the per-center remainders:
//   J = (sum s^2 - sum_j T_j / N_j) 2^-2F + sum_j N_j ||c_j - mu_j||^2
//     = sum_j sum_{i in j} ||x_i - c_j||^2   (Eq. 3, on the fixed-point values).
// Ends with the block synchronised.
static __device__ void finalize_reduce_block(int k, const unsigned long long* cnt, StageState* st,
                                             const TrajDev& tr, const double* clus, FinalizeSmem& sm)
{
    constexpr int B = 256;
    double* traj_J = tr.J;
    double* traj_shift = tr.shift;
    const unsigned long long* qw = reinterpret_cast<const unsigned long long*>(clus + 3 * k);
    const double inv = st->inv_scaleF;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double sh = 0.0, mx = 0.0;
    double jj[4] = {0.0, 0.0, 0.0, 0.0};         // threads tid, tid + 256, .. of the 1024
    int em = 0;
    unsigned __int128 a0 = 0, a1 = 0, a2 = 0;    // sums of the limbs of floor(T_j / N_j)
    for (int j0 = 0; j0 < k; j0 += 1024) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int j = j0 + B * v + tid;
            if (j >= k) break;
            sh = fmax(sh, __ldcg(clus + j));
            mx = fmax(mx, __ldcg(clus + 2 * k + j));
            jj[v] += __ldcg(clus + k + j);
            if (__ldcg(cnt + j) == 0) {
                ++em;
            } else {
                a0 += __ldcg(qw + 3ll * j);
                a1 += __ldcg(qw + 3ll * j + 1);
                a2 += __ldcg(qw + 3ll * j + 2);
            }
        }
    }
    // the 1024-thread tree's first two levels, then 256 values
    sm.r_J[tid] = (jj[0] + jj[2]) + (jj[1] + jj[3]);
    a0 = warp_sum_u128(a0);
    a1 = warp_sum_u128(a1);
    a2 = warp_sum_u128(a2);
    for (int o = 16; o; o >>= 1) {
        sh = fmax(sh, __shfl_xor_sync(0xffffffffu, sh, o));
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        em += __shfl_xor_sync(0xffffffffu, em, o);
    }
    if (lane == 0) {
        sm.r_shift[warp] = sh;
        sm.r_nn[warp] = mx;
        sm.r_empty[warp] = em;
        sm.r_q[warp][0] = a0;
        sm.r_q[warp][1] = a1;
        sm.r_q[warp][2] = a2;
    }
    __syncthreads();
    if (warp == 0) {
        double r[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) r[v] = sm.r_J[lane + 32 * v];
        // levels 128, 64, 32 of the tree in this lane, 16 .. 1 across lanes
        double J0 = ((r[0] + r[4]) + (r[2] + r[6])) + ((r[1] + r[5]) + (r[3] + r[7]));
        for (int o = 16; o; o >>= 1) J0 += __shfl_down_sync(0xffffffffu, J0, o);
        const bool in = lane < B / 32;
        sh = in ? sm.r_shift[lane] : 0.0;
        mx = in ? sm.r_nn[lane] : 0.0;
        em = in ? sm.r_empty[lane] : 0;
        a0 = in ? sm.r_q[lane][0] : (unsigned __int128)0;
        a1 = in ? sm.r_q[lane][1] : (unsigned __int128)0;
        a2 = in ? sm.r_q[lane][2] : (unsigned __int128)0;
        a0 = warp_sum_u128(a0);
        a1 = warp_sum_u128(a1);
        a2 = warp_sum_u128(a2);
        for (int o = 16; o; o >>= 1) {
            sh = fmax(sh, __shfl_xor_sync(0xffffffffu, sh, o));
            mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            em += __shfl_xor_sync(0xffffffffu, em, o);
        }
        if (lane == 0) {
            // D = sum s^2 - sum_j floor(T_j / N_j)  (>= 0: Cauchy-Schwarz per cluster)
            U256 D = {{0ull, 0ull, 0ull, 0ull}};
            U256 Tq = {{0ull, 0ull, 0ull, 0ull}};
            u256_add_at(D, (unsigned __int128)st->q[0], 0);
            u256_add_at(D, (unsigned __int128)st->q[1] << 32, 0);
            u256_add_at(D, (unsigned __int128)st->q[2], 1);
            u256_add_at(D, (unsigned __int128)st->q[3] << 32, 1);
            u256_add_at(Tq, a0, 0);
            u256_add_at(Tq, a1, 1);
            u256_add_at(Tq, a2, 2);
            u256_neg(Tq);
            for (int i = 0; i < 4; ++i) u256_add_at(D, (unsigned __int128)Tq.w[i], i);
            double J = u256_to_double(D) * (inv * inv) + J0;
            if (J < 0.0) J = 0.0;   // only rounding of an exactly zero objective can go below
            double shift = sqrt(sh);
            int it = st->iter;
            if (traj_J) traj_J[it] = J;
            if (traj_shift) traj_shift[it] = shift;
            st->J = J;
            st->shift = shift;
            st->empty = em;
            st->cmax2 = __double2float_ru(mx);
            st->iter = it + 1;
            int conv = shift <= st->tol;
            st->converged = conv;
            st->done = conv || (it + 1 >= st->max_iter);
            st->mode = kModeDelta;
            st->rechecked_total += st->recheck_count;
            st->listed_total += st->recheck_count;
            st->recheck_count = 0;
        }
    }
    __syncthreads();
}

// FP32 D_j = ||c_j||^2 - 2 x.c_j of one point against centers j0 + 32 i
// (i < NQ): the CUDA-core FMA chain whose error tie_kappa bounds, t ascending.
// c32t (dims x kpad, coalesced across the warp's lanes) holds the same FP32
// values as the row-major copy; fmaf(-2 x_t, c_t, a) equals fmaf(x_t, -2 c_t, a)
// (scaling by -2 is exact).  Padding centers read zeros.
template <int NQ>
static __device__ __forceinline__ void recheck_d(const float* __restrict__ x, int d,
                                                 const Centers& c, int j0, float (&a)[NQ])
{
    const int kpad = c.kpad;
#pragma unroll
    for (int i = 0; i < NQ; ++i) a[i] = c.cnorm[j0 + 32 * i];
    const float* ct = c.c32t + j0;
    int t = 0;
    if ((reinterpret_cast<uintptr_t>(x) & 15) == 0) {
#pragma unroll 2
        for (; t + 4 <= d; t += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(x + t));
            const float xm2[4] = {-2.0f * v.x, -2.0f * v.y, -2.0f * v.z, -2.0f * v.w};
            float w[4][NQ];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int i = 0; i < NQ; ++i) w[u][i] = ct[(long long)(t + u) * kpad + 32 * i];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int i = 0; i < NQ; ++i) a[i] = fmaf(xm2[u], w[u][i], a[i]);
        }
    }
#pragma unroll 4
    for (; t < d; ++t) {
        const float xm2 = -2.0f * __ldg(x + t);
        const float* row = ct + (long long)t * kpad;
#pragma unroll
        for (int i = 0; i < NQ; ++i) a[i] = fmaf(xm2, row[32 * i], a[i]);
    }
}

// The sums, counts and label of point i (row x) move from cluster old (-1: none)
// to bj; threads tid of nt share the coordinates.
static __device__ __forceinline__ void recheck_move(const float* __restrict__ x, int d, const Accum& acc,
                                                    int* __restrict__ labels, int i, int old, int bj,
                                                    float scaleF, int tid, int nt)
{
    for (int t = tid; t < d; t += nt) {
        long long v = to_fixed(__ldg(x + t), scaleF);
        split_add(acc.s_lo + (long long)bj * d + t, acc.s_hi + (long long)bj * d + t, v);
        if (old >= 0)
            split_add(acc.s_lo + (long long)old * d + t, acc.s_hi + (long long)old * d + t, -v);
    }
    if (tid == 0) {
        atomicAdd(acc.cnt + bj, 1ull);
        if (old >= 0) atomicAdd(acc.cnt + old, ~0ull);
        labels[i] = bj;
    }
}

// One warp: FP64 squared distance of row x to center j, lanes over coordinates.
static __device__ __forceinline__ double recheck_lanes_f64(const float* __restrict__ x, int d,
                                                           const Centers& c, int j)
{
    const double* cj64 = c.c64 + (long long)j * d;
    double p = 0.0;
    for (int t = threadIdx.x & 31; t < d; t += 32) {
        const double e = (double)__ldg(x + t) - cj64[t];
        p = fma(e, e, p);
    }
    return warp_sum_f64(p);
}

// Whether the best two of recheck_lanes_f64 rank the same in the oracle's order.
static __device__ __forceinline__ bool recheck_ranked(double s1, double s2, int d)
{
    return s2 - s1 > (double)(2 * d + 16) * 1.1102230246251565e-16 * (s1 + s2);
}

// One warp: re-decide point i.  Pass 1: FP32 D_j for every center on the CUDA
// cores (recheck_d) and their minimum b1.  Pass 2: the centers with D_j <= b1 +
// tie_kappa (2 C2 + X2) + tie_abs -- a set that provably holds the FP64 argmin -- are
// compared by their FP64 distances and the smallest wins, lowest index on ties,
// as in the oracle's form (sum_t fma(x_t - c_t, x_t - c_t, acc), t ascending):
//   one candidate   it is the argmin;
//   few, d > 16     the lanes share a candidate's coordinates: 2 d / 32 + 5 FP64
//                   instructions each, in another order of addition, which
//                   decides when the best two differ by more than both orders'
//                   rounding (d + 7 and d + 1 roundings of 2^-53 at most);
//   otherwise       a lane per candidate in the oracle's order (2 d FP64
//                   instructions).
// An FP64 instruction holds the SM's FP64 pipe for 16 cycles whatever its active
// lanes, so at d = 128 the second form takes 26 instead of 256 pipe slots for a
// pair of candidates (recheck of 8,600 points, k = 32: 82 -> 39 us).
// The point's new label and the sums follow (delta mode: from its old label).
// cache: per-warp shared memory of cache_cap floats for the pass-1 values
// (pass 2 recomputes them when kpad > cache_cap or cache is null).  Returns
// whether the point had a single candidate.
// NQ: centers per lane and step (1 for k <= 32, 2 for k <= 64, else 4).
template <int NQ>
static __device__ __forceinline__ bool recheck_point_nq(const float* __restrict__ X, int d,
                                                        const Centers& c, int* __restrict__ labels,
                                                        int i, StageState* st, const Accum& acc,
                                                        float* cache, int cache_cap)
{
    constexpr int STEP = 32 * NQ;
    const int mode = st->mode;
    const float c2x2 = 2.0f * st->cmax2;
    const float kap = tie_kappa(d);
    const int k = c.k;
    const bool cached = cache != nullptr && c.kpad <= cache_cap;
    const int lane = threadIdx.x & 31;
    const float* x = X + (long long)i * d;
    // the old label's load (a random row of the labels) overlaps the passes
    const int old = (mode == kModeDelta) ? labels[i] : -1;
    float x2 = 0.0f;
    for (int t = lane; t < d; t += 32) { float v = __ldg(x + t); x2 = fmaf(v, v, x2); }
    for (int o = 16; o; o >>= 1) x2 += __shfl_xor_sync(0xffffffffu, x2, o);
    float b1 = INFINITY;
    int b1j = k;
    for (int j0 = lane; j0 < k; j0 += STEP) {
        float a[NQ];
        recheck_d<NQ>(x, d, c, j0, a);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            if (j0 + 32 * q < k && a[q] < b1) { b1 = a[q]; b1j = j0 + 32 * q; }
            if (cached) cache[j0 + 32 * q] = a[q];
        }
    }
    const float lane_b1 = b1;
    for (int o = 16; o; o >>= 1) b1 = fminf(b1, __shfl_xor_sync(0xffffffffu, b1, o));
    const float lim = b1 + kap * (c2x2 + x2) * 1.0009765625f + tie_abs(d + 1);
    auto value = [&](int j0, float (&a)[NQ]) {
        if (cached) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) a[q] = cache[j0 + 32 * q];
        } else {
            recheck_d<NQ>(x, d, c, j0, a);
        }
    };
    int ncand = 0;
    for (int j0 = lane; j0 < k; j0 += STEP) {
        float a[NQ];
        value(j0, a);
#pragma unroll
        for (int q = 0; q < NQ; ++q) ncand += (j0 + 32 * q < k && a[q] <= lim) ? 1 : 0;
    }
    ncand = __reduce_add_sync(0xffffffffu, ncand);
    int bj = INT_MAX;
    bool decided = false;
    const bool single = ncand == 1 && lim < FLT_MAX;
    if (single) {
        const unsigned m = __ballot_sync(0xffffffffu, lane_b1 == b1);
        bj = __shfl_sync(0xffffffffu, b1j, __ffs(m) - 1);
        decided = true;
    } else if (d > 16 && ncand * (2 * ((d + 31) / 32) + 5) < 2 * d) {
        double s1 = DBL_MAX, s2 = DBL_MAX;       // best two sums (the same on every lane)
        for (int jb = 0; jb < k; jb += STEP) {
            float a[NQ];
            if (jb + lane < k) value(jb + lane, a);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                unsigned m = __ballot_sync(0xffffffffu, jb + lane + 32 * q < k && a[q] <= lim);
                while (m) {
                    const int j = jb + 32 * q + __ffs(m) - 1;
                    m &= m - 1;
                    const double p = recheck_lanes_f64(x, d, c, j);
                    if (p < s1) { s2 = s1; s1 = p; bj = j; }
                    else if (p < s2) s2 = p;
                }
            }
        }
        decided = recheck_ranked(s1, s2, d);
    }
    if (!decided) {
        double best = DBL_MAX;
        bj = INT_MAX;
        for (int j0 = lane; j0 < k; j0 += STEP) {
            float a[NQ];
            value(j0, a);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int j = j0 + 32 * q;
                if (j < k && a[q] <= lim) {
                    const double* cj64 = c.c64 + (long long)j * d;
                    double a2 = 0.0;
                    for (int t = 0; t < d; ++t) {
                        double e = (double)__ldg(x + t) - cj64[t];
                        a2 = fma(e, e, a2);
                    }
                    if (a2 < best || (a2 == best && j < bj)) { best = a2; bj = j; }
                }
            }
        }
        // lowest (distance, index) over the lanes; the FP64 sums of squares are
        // non-negative, so their bit patterns order as the values do and the
        // comparison stays off the (narrow) FP64 pipe
        unsigned long long bb = (unsigned long long)__double_as_longlong(best);
        for (int o = 16; o; o >>= 1) {
            const unsigned long long ob = __shfl_xor_sync(0xffffffffu, bb, o);
            const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
            if (ob < bb || (ob == bb && oj < bj)) { bb = ob; bj = oj; }
        }
    }
    __syncwarp();   // every lane has read the old label before lane 0 rewrites it
    if (bj != old && label_ok(bj, k, st) && old_label_ok(old, k, st))
        recheck_move(x, d, acc, labels, i, old, bj, st->scaleF, lane, 32);
    return single;
}

static __device__ __forceinline__ bool recheck_point(const float* __restrict__ X, int d,
                                                     const Centers& c, int* __restrict__ labels,
                                                     int i, StageState* st, const Accum& acc,
                                                     float* cache, int cache_cap)
{
    if (c.k <= 32) return recheck_point_nq<1>(X, d, c, labels, i, st, acc, cache, cache_cap);
    if (c.k <= 64) return recheck_point_nq<2>(X, d, c, labels, i, st, acc, cache, cache_cap);
    return recheck_point_nq<4>(X, d, c, labels, i, st, acc, cache, cache_cap);
}

// The same for more centers than the cache holds values of: pass 2 forms the values
// again, once, and the candidates' indices (ascending) take the cache, cap of them;
// a point with more is compared in a third pass.  (Counting the candidates and then
// comparing them formed the values three or four times: a step of 1e6 x 2, k = 20,000 at
// an offset of 100 74.6 ms, now 45.1; 5e5 x 17, k = 1,025 3.3 and 2.5.)
static __device__ __forceinline__ bool recheck_point_large(const float* __restrict__ X, int d, const Centers& c,
                                                        int* __restrict__ labels, int i, StageState* st,
                                                        const Accum& acc, int* cand, int cap)
{
    constexpr int NQ = 4, STEP = 32 * NQ;
    const int k = c.k, lane = threadIdx.x & 31;
    const float* x = X + (long long)i * d;
    const int old = (st->mode == kModeDelta) ? labels[i] : -1;
    float x2 = 0.0f;
    for (int t = lane; t < d; t += 32) { float v = __ldg(x + t); x2 = fmaf(v, v, x2); }
    for (int o = 16; o; o >>= 1) x2 += __shfl_xor_sync(0xffffffffu, x2, o);
    // recheck_d without its vector loads' tests, which outweigh the products for d < 4
    auto value = [&](int j0, float (&a)[NQ]) {
        if (d >= 4) {
            recheck_d<NQ>(x, d, c, j0, a);
            return;
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) a[q] = c.cnorm[j0 + 32 * q];
#pragma unroll 1
        for (int t = 0; t < d; ++t) {
            const float xm2 = -2.0f * __ldg(x + t);
            const float* row = c.c32t + (long long)t * c.kpad + j0;
#pragma unroll
            for (int q = 0; q < NQ; ++q) a[q] = fmaf(xm2, row[32 * q], a[q]);
        }
    };
    float b1 = INFINITY;
    // (kpad is a multiple of STEP; padding centers read as FLT_MAX)
    for (int j0 = lane; j0 < c.kpad; j0 += STEP) {
        float a[NQ];
        value(j0, a);
        b1 = fmin3(b1, a[0], a[1]);
        b1 = fmin3(b1, a[2], a[3]);
    }
    for (int o = 16; o; o >>= 1) b1 = fminf(b1, __shfl_xor_sync(0xffffffffu, b1, o));
    const float lim = b1 + tie_kappa(d) * (2.0f * st->cmax2 + x2) * 1.0009765625f + tie_abs(d + 1);
    int ncand = 0;
    for (int j0 = lane; j0 < c.kpad; j0 += STEP) {
        float a[NQ];
        value(j0, a);
        if (!__any_sync(0xffffffffu, a[0] <= lim || a[1] <= lim || a[2] <= lim || a[3] <= lim)) continue;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const bool near = j0 + 32 * q < k && a[q] <= lim;
            const unsigned m = __ballot_sync(0xffffffffu, near);
            const int at = ncand + __popc(m & lanemask_lt());
            if (near && at < cap) cand[at] = j0 + 32 * q;
            ncand += __popc(m);
        }
    }
    __syncwarp();
    int bj = INT_MAX;
    bool decided = false;
    const bool single = ncand == 1 && lim < FLT_MAX;
    if (single) {
        bj = cand[0];
        decided = true;
    } else if (d > 16 && ncand <= cap && ncand * (2 * ((d + 31) / 32) + 5) < 2 * d) {
        double s1 = DBL_MAX, s2 = DBL_MAX;
        for (int e = 0; e < ncand; ++e) {
            const int j = cand[e];
            const double p = recheck_lanes_f64(x, d, c, j);
            if (p < s1) { s2 = s1; s1 = p; bj = j; }
            else if (p < s2) s2 = p;
        }
        decided = recheck_ranked(s1, s2, d);
    }
    if (!decided) {
        double best = DBL_MAX;
        bj = INT_MAX;
        auto compare = [&](int j) {
            const double* cj64 = c.c64 + (long long)j * d;
            double a2 = 0.0;
            for (int t = 0; t < d; ++t) {
                double e = (double)__ldg(x + t) - cj64[t];
                a2 = fma(e, e, a2);
            }
            if (a2 < best || (a2 == best && j < bj)) { best = a2; bj = j; }
        };
        if (ncand <= cap) {
            for (int e = lane; e < ncand; e += 32) compare(cand[e]);
        } else {
            for (int j0 = lane; j0 < k; j0 += STEP) {
                float a[NQ];
                value(j0, a);
#pragma unroll
                for (int q = 0; q < NQ; ++q)
                    if (j0 + 32 * q < k && a[q] <= lim) compare(j0 + 32 * q);
            }
        }
        unsigned long long bb = (unsigned long long)__double_as_longlong(best);
        for (int o = 16; o; o >>= 1) {
            const unsigned long long ob = __shfl_xor_sync(0xffffffffu, bb, o);
            const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
            if (ob < bb || (ob == bb && oj < bj)) { bb = ob; bj = oj; }
        }
    }
    __syncwarp();   // every lane has read the old label and the candidates
    if (bj != old && label_ok(bj, k, st) && old_label_ok(old, k, st))
        recheck_move(x, d, acc, labels, i, old, bj, st->scaleF, lane, 32);
    return single;
}

// A block of 256 threads per point, for many centers and few listed points: the
// warps share the centers, so a point waits for an eighth of the loads (one warp
// per point is bound by their latency: k = 1024, d = 128 reads 512 KB of centers).
// The same decisions as recheck_point.  cache: kpad floats of shared memory.
struct RecheckBlockSmem {
    float b1[8];
    int b1j[8];
    int ncand[8];
    double s1[8], s2[8];
    int sj[8];
    int bj;
};
static __device__ bool recheck_point_block(const float* __restrict__ X, int d, const Centers& c,
                                           int* __restrict__ labels, int i, StageState* st,
                                           const Accum& acc, float* cache, RecheckBlockSmem& sm)
{
    const int k = c.k;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float* x = X + (long long)i * d;
    const int old = (st->mode == kModeDelta) ? labels[i] : -1;
    float x2 = 0.0f;
    for (int t = lane; t < d; t += 32) { float v = __ldg(x + t); x2 = fmaf(v, v, x2); }
    for (int o = 16; o; o >>= 1) x2 += __shfl_xor_sync(0xffffffffu, x2, o);
    float b1 = INFINITY;
    int b1j = k;
    for (int j0 = 32 * warp + lane; j0 < k; j0 += 256) {
        float a[1];
        recheck_d<1>(x, d, c, j0, a);
        if (a[0] < b1) { b1 = a[0]; b1j = j0; }
        cache[j0] = a[0];
    }
    const float lane_b1 = b1;
    for (int o = 16; o; o >>= 1) b1 = fminf(b1, __shfl_xor_sync(0xffffffffu, b1, o));
    {
        const unsigned m = __ballot_sync(0xffffffffu, lane_b1 == b1);
        b1j = __shfl_sync(0xffffffffu, b1j, m ? __ffs(m) - 1 : 0);
    }
    if (lane == 0) { sm.b1[warp] = b1; sm.b1j[warp] = b1j; }
    __syncthreads();
    int bj = INT_MAX;
    for (int w = 0; w < 8; ++w)
        if (sm.b1[w] < b1 || (sm.b1[w] == b1 && w <= warp)) b1 = sm.b1[w];
    for (int w = 7; w >= 0; --w)
        if (sm.b1[w] == b1) bj = sm.b1j[w];
    const float lim = b1 + tie_kappa(d) * (2.0f * st->cmax2 + x2) * 1.0009765625f + tie_abs(d + 1);
    int nc = 0;
    double s1 = DBL_MAX, s2 = DBL_MAX;
    int sj = INT_MAX;
    for (int jb = 32 * warp; jb < k; jb += 256) {
        unsigned m = __ballot_sync(0xffffffffu, jb + lane < k && cache[jb + lane] <= lim);
        nc += __popc(m);
    }
    if (lane == 0) sm.ncand[warp] = nc;
    __syncthreads();
    int ncand = 0;
    for (int w = 0; w < 8; ++w) ncand += sm.ncand[w];
    const bool single = ncand == 1 && lim < FLT_MAX;
    bool decided = single;
    if (!single && ncand <= 256) {
        for (int jb = 32 * warp; jb < k; jb += 256) {
            unsigned m = __ballot_sync(0xffffffffu, jb + lane < k && cache[jb + lane] <= lim);
            while (m) {
                const int j = jb + __ffs(m) - 1;
                m &= m - 1;
                const double p = recheck_lanes_f64(x, d, c, j);
                if (p < s1) { s2 = s1; s1 = p; sj = j; }
                else if (p < s2) s2 = p;
            }
        }
        if (lane == 0) { sm.s1[warp] = s1; sm.s2[warp] = s2; sm.sj[warp] = sj; }
        __syncthreads();
        s1 = s2 = DBL_MAX;
        bj = INT_MAX;
        for (int w = 0; w < 8; ++w) {
            const double a1 = sm.s1[w], a2 = sm.s2[w];
            if (a1 < s1) { s2 = fmin(s1, a2); s1 = a1; bj = sm.sj[w]; }
            else s2 = fmin(s2, a1);
        }
        decided = recheck_ranked(s1, s2, d);
    }
    if (!decided) {                              // the same on every thread
        if (warp == 0) {
            // the oracle's order, a lane per candidate
            double best = DBL_MAX;
            bj = INT_MAX;
            for (int j = lane; j < k; j += 32) {
                if (cache[j] <= lim) {
                    const double* cj64 = c.c64 + (long long)j * d;
                    double a2 = 0.0;
                    for (int t = 0; t < d; ++t) {
                        double e = (double)__ldg(x + t) - cj64[t];
                        a2 = fma(e, e, a2);
                    }
                    if (a2 < best || (a2 == best && j < bj)) { best = a2; bj = j; }
                }
            }
            unsigned long long bb = (unsigned long long)__double_as_longlong(best);
            for (int o = 16; o; o >>= 1) {
                const unsigned long long ob = __shfl_xor_sync(0xffffffffu, bb, o);
                const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
                if (ob < bb || (ob == bb && oj < bj)) { bb = ob; bj = oj; }
            }
            if (lane == 0) sm.bj = bj;
        }
        __syncthreads();
        bj = sm.bj;
    }
    __syncthreads();   // every thread has read the old label and the shared values
    if (bj != old && label_ok(bj, k, st) && old_label_ok(old, k, st))
        recheck_move(x, d, acc, labels, i, old, bj, st->scaleF, threadIdx.x, blockDim.x);
    return single;
}

// One warp per listed point; warps gw, gw + nw, ... of the caller each take the
// listed points.  cache: cache_cap floats per warp (LARGE: kpad is above it).
// settles: the list comes from a screen that leaves rows to the FP32 pass here;
// those it decides alone do not count as rechecked in FP64.
template <bool LARGE>
static __device__ void recheck_warps(const float* __restrict__ X, int d, Centers c,
                                     int* __restrict__ labels, const int* __restrict__ list,
                                     StageState* st, Accum acc, long long gw, long long nw,
                                     float* cache, int cache_cap, int settles)
{
    const int count = st->recheck_count;
    long long settled = 0;
    for (long long w = gw; w < count; w += nw) {
        if constexpr (LARGE)
            settled += recheck_point_large(X, d, c, labels, list[w], st, acc, reinterpret_cast<int*>(cache),
                                           cache_cap) ? 1 : 0;
        else
            settled += recheck_point(X, d, c, labels, list[w], st, acc, cache, cache_cap) ? 1 : 0;
    }
    if (settles && settled && (threadIdx.x & 31) == 0)
        atomicAdd(reinterpret_cast<unsigned long long*>(&st->rechecked_total),
                  (unsigned long long)(-settled));
}


}  // namespace km2
