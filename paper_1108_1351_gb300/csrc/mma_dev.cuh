// mma_dev.cuh -- warp-level distance core of the tensor-core screen: one warp
// decides 32 rows against k centers from split-FP16 products on mma.sync
// (assign_mma.cu and batched.cu run it; recheck_fp32_row settles what it
// leaves open).
//
// Key of center j for a row x, in scaled units (S = sx sm, powers of two):
//   key_j = sum_t xs_t ms_jt + S ||c_j||^2,  xs = sx x, ms = -2 sm c_j,
// each operand split into two FP16 parts (hi + lo, 22 significant bits), the
// products accumulated in FP32 by the tensor core with the small (lo) terms
// first, and the FP32 norm added last, so the accumulator never holds a value of
// the norm's size.  A row whose best key is separated from every other by more
// than mma_thr's bound is decided here: its argmin is the exact one.  Any other
// row is decided again on the CUDA cores with the FP32 FMA chain and that chain's
// bound (tie_kappa), and what that leaves open goes to the FP64 recheck, so labels
// equal those of every other form bit for bit.
//
// Keys are no less precise than the FP32 chain's from d = 8 on.  Error against
// FP64, rms / largest, in 2^-24 (||x||^2 + 2 C^2), isotropic and anisotropic
// mixtures of 50 components: d = 8 0.26 / 1.9 (chain 0.27 / 2.1), d = 12 0.27 / 1.9
// (0.33 / 2.9), d = 16 0.25 / 1.7 (0.39 / 3.0), d = 32 0.26 / 2.5 (0.56 / 3.5), d = 64 0.37
// / 4.4 (0.80 / 4.9), d = 128 0.34 / 4.1 (1.19 / 6.1); largest error 0.02 of the bound.
// Below, two parts are less precise (d = 4 0.35, chain 0.24) and a third part costs
// what the MMAs save (n = 1e7, d = 4, k = 20: 135 us against 121), so d < 8 stays on
// the CUDA cores.
//
// Why tensor cores here: at d = 8 the CUDA-core loop spends 8 FMA cycles and
// ~7 ALU cycles per 32 distances and they hardly overlap (16-20 cycles
// measured).  The two m16n8k16 MMAs of a 16 x 8 block cost 4 cycles per 32
// distances, and the selection ~3.5: a 3-input minimum (2 cycles, two keys),
// a packed add of the norm and one of the bound, and a funnel shift (2 cycles)
// that collects the sign of key - (minimum + bound); the packed-key top-2 took
// ~7.  Measured rates (cycles per warp instruction and SM sub-partition): MMA 8,
// FFMA / FADD 1, packed FP32x2 2, minimum / logic / shift 2, shuffle 4; MMAs and
// FFMAs do not overlap (both wait for register ports), MMAs and ALU work half.
//
// Fragment layout (m16n8k16): lane = 4 g + t holds rows g and g + 8 of a
// 16-row block and columns 2 t, 2 t + 1 of an 8-center block.  A warp holds
// two row blocks, so a lane has four row slots s = 2 (block) + (row >= 8): slot
// s is row 8 s + g of the 32.  After the scan lane (g, t) owns row 8 t + g.
// Coordinates may be assigned to the K slots in any order that A and B share:
//   DP = 8   slot pair t holds dims 2 t, 2 t + 1; [xh | xl] x [ml | ml], then
//            [xh | xl] x [mh | mh]
//   DP = 16 KS  K-step ks, lane t: dims 16 ks + 4 t .. + 3 (one 128-bit read
//            per row); xl mh and xh ml of all K-steps, then xh mh
#pragma once

#include <cfloat>

#include <cuda_fp16.h>

#include "common.cuh"

namespace km2 {

template <int DP>
struct MmaCfg {
    static constexpr int KS = DP >= 16 ? DP / 16 : 1;         // K-steps
    static constexpr int AREG = DP >= 16 ? 8 * KS : 4;        // A registers per row block
    static constexpr int BW = 4 * KS;                         // B words per lane and 8 centers
};

// Bytes of the centers' fragments per 8-center block, and of their norms.
__host__ __device__ constexpr int mma_bw(int dp) { return dp >= 16 ? dp / 4 : 4; }
__host__ __device__ inline size_t mma_center_bytes(int dp, int ntiles)
{
    return (size_t)ntiles * (mma_bw(dp) * 128 + 32);
}
__host__ __device__ inline int mma_dp(int d)
{
    return d <= 8 ? 8 : d <= 16 ? 16 : d <= 32 ? 32 : d <= 48 ? 48 : d <= 64 ? 64 : d <= 96 ? 96 : 128;
}

// Scales and bound of one pass, derived from the stage state by every CTA.
struct MmaScale {
    float sx, sm, S;     // powers of two; S = sx sm
    // bound = thr0 + thrx * (largest coordinate of the 32 rows)^2;
    // infinite (every row is left open) for centers the scaling does not cover
    float thr0, thrx;
};

// Relative error of a key, in units of (||x||^2 + 2 C^2), for two keys:
//   representation 2 * 2^-22, the dropped xl ml term 2^-22 (DP >= 16), FP32
//   centers and norm, the norm's addition and the comparison's roundings; and
//   the tensor core's accumulation: 17 addends per MMA, each taken as losing
//   2^-23 of the largest magnitude in the sum, over the KS MMAs of the hi
//   products (the lo MMAs run first at 2^-11 of that magnitude or less).
__host__ __device__ inline float mma_kappa(int ks)
{
    return 2.0f * 1.0625f * 1.1920928955078125e-7f * (float)(17 * ks + 12);
}

__device__ __forceinline__ MmaScale mma_scale(const StageState* st, int d, int ks)
{
    MmaScale r;
    const float mx = __uint_as_float(st->maxabs_bits);
    const float c2 = st->cmax2;
    int E = 0, em = 0;
    // exponents below -45 are clamped: S stays finite, and the FP16 subnormal
    // term of the bound takes over as the operands leave the range
    if (mx > 0.0f) { frexpf(mx, &E); E = max(E, -45); }              // max |x| < 2^E
    bool covered = c2 < 1.0e30f && E <= 50;
    if (covered && c2 > 0.0f) {
        frexpf(2.0f * sqrtf(c2), &em);
        em = max(em + 1, -45);                                       // max |2 c| < 2^em
        covered = em - E <= 38;                                      // keys stay below 2^66
    }
    if (!covered) { E = 0; em = 0; }
    r.sx = ldexpf(1.0f, 14 - E);
    r.sm = ldexpf(1.0f, 14 - em);
    r.S = r.sx * r.sm;
    const float kap = mma_kappa(ks);
    // FP16 subnormals: each part is off by up to 2^-25 in scaled units where
    // its relative error is below that, against factors below 2^14
    const float kabs = (float)d * 0.00390625f;
    r.thr0 = covered ? 2.0f * kap * c2 * r.S + kabs + tie_abs(17 * ks + d + 4) * r.S : INFINITY;
    r.thrx = kap * (float)d * r.S;                                   // ||x||^2 <= d max_t x_t^2
    return r;
}

__device__ __forceinline__ void mma16816(float* c, uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
                 "{%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// the same with a zero accumulator
__device__ __forceinline__ void mma16816z(float* c, uint32_t a0, uint32_t a1, uint32_t a2,
                                          uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
                 "{%8,%9}, {%10,%10,%10,%10};"
                 : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.0f));
}
// hi and lo FP16 parts of a pair of scaled values.
__device__ __forceinline__ void split2(float2 v, uint32_t& hi, uint32_t& lo)
{
    const __half2 h = __float22half2_rn(v);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(v.x - f.x, v.y - f.y);   // the differences are exact
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

// The centers' fragments (B operand) into shared memory: sb holds BW words per
// (8-center block, lane) -- for DP >= 16 the hi pairs of every (block, K-step,
// lane) and then the lo pairs -- and sn the scaled norms.  Whole block.
template <int DP>
__device__ __forceinline__ void mma_load_centers(const Centers& c, int ntiles, const MmaScale& ms,
                                                 uint32_t* sb, float* sn)
{
    constexpr int KS = MmaCfg<DP>::KS;
    const int k = c.k, d = c.d;
    auto val = [&](int j, int t) -> float {
        return (j < k && t < d) ? -2.0f * c.c32[(long long)j * d + t] * ms.sm : 0.0f;
    };
    for (int e = threadIdx.x; e < ntiles * KS * 32; e += blockDim.x) {
        const int lane = e & 31, g = lane >> 2, t = lane & 3;
        const int ks = (e >> 5) % KS, nt = (e >> 5) / KS;
        const int j = nt * 8 + g;
        uint32_t hi, lo;
        if constexpr (DP >= 16) {
            uint32_t hi2, lo2;
            split2(make_float2(val(j, 16 * ks + 4 * t), val(j, 16 * ks + 4 * t + 1)), hi, lo);
            split2(make_float2(val(j, 16 * ks + 4 * t + 2), val(j, 16 * ks + 4 * t + 3)), hi2, lo2);
            reinterpret_cast<uint2*>(sb)[e] = make_uint2(hi, hi2);
            reinterpret_cast<uint2*>(sb)[ntiles * KS * 32 + e] = make_uint2(lo, lo2);
        } else {
            split2(make_float2(val(j, 2 * t), val(j, 2 * t + 1)), hi, lo);
            // both B registers of an MMA hold the same pair: stored twice, so
            // that one 128-bit load yields register pairs
            reinterpret_cast<uint4*>(sb)[e] = make_uint4(hi, hi, lo, lo);
        }
    }
    for (int j = threadIdx.x; j < ntiles * 8; j += blockDim.x)
        sn[j] = j < k ? c.cnorm[j] * ms.S : FLT_MAX;      // padding: never the best
}

// A registers of the lane's two rows of a 16-row block from 32 rows of d floats
// (shared memory), and the running maximum of the coordinates' magnitudes.
// FULL: d == DP.
template <int DP, bool FULL>
__device__ __forceinline__ void mma_load_rows(const float* xr, int d, int g, int t, int blk, float sx,
                                              uint32_t* A, float& xmax)
{
    constexpr int KS = MmaCfg<DP>::KS;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float* p = xr + (blk * 16 + h * 8 + g) * (FULL ? DP : d);
        if constexpr (DP >= 16) {
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                const int t0 = 16 * ks + 4 * t;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (FULL) {
                    v = *reinterpret_cast<const float4*>(p + t0);
                } else if ((d & 3) == 0) {
                    if (t0 < d) v = *reinterpret_cast<const float4*>(p + t0);
                } else {
                    if (t0 < d) v.x = p[t0];
                    if (t0 + 1 < d) v.y = p[t0 + 1];
                    if (t0 + 2 < d) v.z = p[t0 + 2];
                    if (t0 + 3 < d) v.w = p[t0 + 3];
                }
                // A[8 ks + ..]: hi {a0, a1, a2, a3}, lo {a0, a1, a2, a3}
                split2(make_float2(v.x * sx, v.y * sx), A[8 * ks + h], A[8 * ks + 4 + h]);
                split2(make_float2(v.z * sx, v.w * sx), A[8 * ks + 2 + h], A[8 * ks + 6 + h]);
                xmax = fmaxf(fmaxf(xmax, fabsf(v.x)), fabsf(v.y));
                xmax = fmaxf(fmaxf(xmax, fabsf(v.z)), fabsf(v.w));
            }
        } else {
            // d == 8
            const float2 v = *reinterpret_cast<const float2*>(p + 2 * t);
            split2(make_float2(v.x * sx, v.y * sx), A[h], A[2 + h]);
            xmax = fmaxf(fmaxf(xmax, fabsf(v.x)), fabsf(v.y));
        }
    }
}

// The bound of the warp's 32 rows from the lanes' maxima (non-negative floats
// order as their bits).
__device__ __forceinline__ float mma_thr(const MmaScale& ms, float xmax)
{
    const float f = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(xmax)));
    return fmaf(ms.thrx * f, f, ms.thr0);
}

// Keys without the norm of both row blocks against NT 8-center blocks.
template <int DP, int NT>
__device__ __forceinline__ void mma_chunk(const uint32_t (&A)[2][MmaCfg<DP>::AREG], const uint32_t* sb,
                                          int nt0, int ntiles, int lane, float (&acc)[2][NT][4])
{
    constexpr int KS = MmaCfg<DP>::KS;
    if constexpr (DP >= 16) {
        const uint2* bh = reinterpret_cast<const uint2*>(sb) + (size_t)nt0 * KS * 32 + lane;
        const uint2* bl = bh + (size_t)ntiles * KS * 32;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
#pragma unroll
            for (int q = 0; q < NT; ++q) {
                const uint2 h = bh[(q * KS + ks) * 32], l = bl[(q * KS + ks) * 32];
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const uint32_t* a = A[b] + 8 * ks;
                    if (ks == 0) mma16816z(acc[b][q], a[0], a[1], a[2], a[3], l.x, l.y);
                    else mma16816(acc[b][q], a[0], a[1], a[2], a[3], l.x, l.y);
                    mma16816(acc[b][q], a[4], a[5], a[6], a[7], h.x, h.y);
                    if (KS == 1) mma16816(acc[b][q], a[0], a[1], a[2], a[3], h.x, h.y);
                }
            }
        }
        if constexpr (KS > 1) {
            // from six K-steps on the hi products go to two accumulators, added in
            // FP32: half the truncations at half the magnitude (d = 128: largest key
            // error 7.7 in one accumulator, 6.4 for the FP32 chain)
            constexpr bool TWO = KS > 4;
            float acc2[2][TWO ? NT : 1][4];
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
#pragma unroll
                for (int q = 0; q < NT; ++q) {
                    const uint2 h = bh[(q * KS + ks) * 32];
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                        const uint32_t* a = A[b] + 8 * ks;
                        if (TWO && ks == 0) mma16816z(acc2[b][q], a[0], a[1], a[2], a[3], h.x, h.y);
                        else if (TWO && ks < KS / 2) mma16816(acc2[b][q], a[0], a[1], a[2], a[3], h.x, h.y);
                        else mma16816(acc[b][q], a[0], a[1], a[2], a[3], h.x, h.y);
                    }
                }
            }
            if constexpr (TWO) {
#pragma unroll
                for (int b = 0; b < 2; ++b)
#pragma unroll
                    for (int q = 0; q < NT; ++q)
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[b][q][e] += acc2[b][q][e];
            }
        }
    } else {
        const uint4* bp = reinterpret_cast<const uint4*>(sb) + (size_t)nt0 * 32 + lane;
#pragma unroll
        for (int q = 0; q < NT; ++q) {
            const uint4 w = bp[q * 32];
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                mma16816z(acc[b][q], A[b][0], A[b][1], A[b][2], A[b][3], w.z, w.w);
                mma16816(acc[b][q], A[b][0], A[b][1], A[b][2], A[b][3], w.x, w.y);
            }
        }
    }
}

__device__ __forceinline__ uint32_t shf_sign(float t, uint32_t m)
{
    return __funnelshift_l(__float_as_uint(t), m, 1);     // (m << 1) | sign(t)
}

// 4 x 4 transpose across a quad: afterwards v[i] is what lane t ^ i of the quad
// held for this lane's slot t.
__device__ __forceinline__ void quad_transpose(uint32_t (&v)[4], int t)
{
    const bool o1 = t & 1, o2 = t & 2;
    const uint32_t a0 = o1 ? v[1] : v[0], s0 = o1 ? v[0] : v[1];
    const uint32_t a1 = o1 ? v[3] : v[2], s1 = o1 ? v[2] : v[3];
    const uint32_t r0 = __shfl_xor_sync(0xffffffffu, s0, 1);
    const uint32_t r1 = __shfl_xor_sync(0xffffffffu, s1, 1);
    v[0] = o2 ? a1 : a0;
    v[1] = o2 ? r1 : r0;
    v[2] = __shfl_xor_sync(0xffffffffu, o2 ? a0 : a1, 2);
    v[3] = __shfl_xor_sync(0xffffffffu, o2 ? r0 : r1, 2);
}

// Decides 32 rows (A: both row blocks) against ntiles 8-center blocks (a
// multiple of NT): the center of the row this lane owns (row 8 t + g), or
// open = true when not exactly one center lies within thr of the best.
// SINGLE: all centers in one chunk of NT blocks (NT <= 4).
template <int DP, int NT, bool SINGLE>
__device__ __forceinline__ int mma_decide(const uint32_t (&A)[2][MmaCfg<DP>::AREG],
                                          const uint32_t* sb, const float* sn, int ntiles, int lane,
                                          float thr, bool& open)
{
    const int t = lane & 3;
    constexpr int NK = 2 * NT;                  // keys per slot and chunk
    float B1[4], B2[4];
    uint32_t MC[4];                             // first block << NK | candidates of the best chunk
    if constexpr (!SINGLE) {
#pragma unroll
        for (int s = 0; s < 4; ++s) { B1[s] = INFINITY; B2[s] = INFINITY; MC[s] = 0; }
    }
    for (int nt0 = 0; nt0 < (SINGLE ? NT : ntiles); nt0 += NT) {
        float acc[2][NT][4];
        mma_chunk<DP, NT>(A, sb, nt0, ntiles, lane, acc);
        float2 nn[NT];
#pragma unroll
        for (int q = 0; q < NT; ++q)
            nn[q] = *reinterpret_cast<const float2*>(sn + (nt0 + q) * 8 + 2 * t);
        uint32_t wall = 0;                      // SINGLE: the slots' masks, one byte each
#pragma unroll
        for (int s = 3; s >= 0; --s) {
            float2 key[NT];
#pragma unroll
            for (int q = 0; q < NT; ++q)
                key[q] = __fadd2_rn(make_float2(acc[s >> 1][q][2 * (s & 1)], acc[s >> 1][q][2 * (s & 1) + 1]), nn[q]);
            float m = fminf(key[0].x, key[0].y);
#pragma unroll
            for (int q = 1; q < NT; ++q) m = fmin3(m, key[q].x, key[q].y);
            const float nT = -(m + thr);
            uint32_t w = SINGLE ? wall << (8 - NK) : (uint32_t)nt0;
#pragma unroll
            for (int q = 0; q < NT; ++q) {
                const float2 v = __fadd2_rn(key[q], make_float2(nT, nT));
                w = shf_sign(v.x, w);
                w = shf_sign(v.y, w);
            }
            if constexpr (SINGLE) {
                B1[s] = m;
                wall = w;
                if (s == 0) MC[0] = w;
            } else {
                if (m < B1[s]) MC[s] = w;
                B2[s] = fminf(B2[s], fmaxf(B1[s], m));
                B1[s] = fminf(B1[s], m);
            }
        }
    }
    // owner lanes: the four column groups of a row side by side
    uint32_t bv[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) bv[s] = __float_as_uint(B1[s]);
    quad_transpose(bv, t);
    const float v0 = __uint_as_float(bv[0]), v1 = __uint_as_float(bv[1]);
    const float v2 = __uint_as_float(bv[2]), v3 = __uint_as_float(bv[3]);
    const float T = fminf(fmin3(v0, v1, v2), v3) + thr;
    if constexpr (SINGLE) {
        // the four masks of at most 8 bits travel as the bytes of one word
        // (byte i from lane t ^ i)
        uint32_t w = MC[0];
        const uint32_t x = __shfl_xor_sync(0xffffffffu, w, 1);
        w = __byte_perm(w, x, (t & 1) ? 0x7351 : 0x6240);
        const uint32_t y = __shfl_xor_sync(0xffffffffu, w, 2);
        w = __byte_perm(w, y, (t & 2) ? 0x7632 : 0x5410);
        if (!(v0 <= T)) w &= 0xffffff00u;
        if (!(v1 <= T)) w &= 0xffff00ffu;
        if (!(v2 <= T)) w &= 0xff00ffffu;
        if (!(v3 <= T)) w &= 0x00ffffffu;
        open = __popc(w) != 1;
        const uint32_t p = (31 - __clz((int)w)) ^ (NK - 1);     // lane << 3 | key index
        return (int)(((p & 6u) << 2) | ((((p >> 3) ^ (uint32_t)t) & 3u) << 1) | (p & 1u));
    } else {
        // another chunk comes close: no valid candidate set
#pragma unroll
        for (int s = 0; s < 4; ++s)
            if (!(B2[s] > B1[s] + thr)) MC[s] = 0;
        quad_transpose(MC, t);
        int cnt = 0, lab = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (__uint_as_float(bv[i]) <= T) {
                const uint32_t cand = MC[i] & ((1u << NK) - 1u);
                cnt += (cand != 0 && (cand & (cand - 1)) == 0) ? 1 : 2;
                const int e = NK - 1 - (31 - __clz((int)cand));
                lab = ((int)(MC[i] >> NK) + (e >> 1)) * 8 + 2 * (i ^ t) + (e & 1);
            }
        }
        open = cnt != 1;
        return lab;
    }
}

// One warp: row x (global) decided with the FP32 FMA chain over all centers
// (recheck_d's values), as the CUDA-core kernels do.  Returns the center, or
// open = true when the best two are within the FP32 bound.
__device__ __forceinline__ int decide_fp32_row(const float* __restrict__ x, int d, const Centers& c,
                                               float thr_base, bool& open)
{
    const int lane = threadIdx.x & 31;
    const int k = c.k, kpad = c.kpad;
    float x2 = 0.0f;
    for (int t = lane; t < d; t += 32) { const float v = __ldg(x + t); x2 = fmaf(v, v, x2); }
    for (int o = 16; o; o >>= 1) x2 += __shfl_xor_sync(0xffffffffu, x2, o);
    float b1 = INFINITY, b2 = INFINITY;
    int bi = 0;
    for (int j0 = lane; j0 < k; j0 += 64) {
        const int j1 = j0 + 32;
        const bool two = j1 < kpad;
        float a0 = c.cnorm[j0], a1 = two ? c.cnorm[j1] : FLT_MAX;
        const float* ct = c.c32t + j0;
#pragma unroll 4
        for (int t = 0; t < d; ++t) {
            const float xm2 = -2.0f * __ldg(x + t);
            a0 = fmaf(xm2, ct[(long long)t * kpad], a0);
            if (two) a1 = fmaf(xm2, ct[(long long)t * kpad + 32], a1);
        }
        if (a0 < b1) { b2 = b1; b1 = a0; bi = j0; } else b2 = fminf(b2, a0);
        if (j1 < k) {
            if (a1 < b1) { b2 = b1; b1 = a1; bi = j1; } else b2 = fminf(b2, a1);
        }
    }
    for (int o = 16; o; o >>= 1) {
        const float o1 = __shfl_xor_sync(0xffffffffu, b1, o);
        const float o2 = __shfl_xor_sync(0xffffffffu, b2, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (o1 < b1 || (o1 == b1 && oi < bi)) { b2 = fminf(b1, o2); b1 = o1; bi = oi; }
        else b2 = fminf(b2, o1);
    }
    // NaN-safe: anything but a provable gap is open
    open = !(b2 - b1 > tie_kappa(d) * (thr_base + x2) + tie_abs(d + 1));
    return bi;
}

// The same for 32 rows at once, a lane per row (x: this lane's row, shared or
// global): what a unit with many open rows takes.  Data far from the origin has
// units in which nearly all rows are open, and row after row they cost up to six
// times what the CUDA-core kernels take for them (a step with an offset of 1000 in
// the data, us, row by row / a lane per row / on CUDA cores: n = 1e6, d = 16, k = 1000
// 7908 / 4116 / 3373, n = 4e6, d = 8, k = 32 2249 / 1623 / 1712).  Bound by FMAs and the
// broadcast loads of the centers.  Returns the center, or -1 for open.
template <int DP, bool FULL>
__device__ __forceinline__ int decide_fp32_lanes(const float* x, int d, const float* __restrict__ cnorm,
                                              const float* __restrict__ c32t, int kpad, int k, float thr_base)
{
    static_assert(DP <= 16, "the row is held in registers");
    float xm2[DP];
    float x2 = 0.0f;
#pragma unroll
    for (int t = 0; t < DP; t += 4) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (FULL) {
            v = *reinterpret_cast<const float4*>(x + t);
        } else {
            if (t < d) v.x = x[t];
            if (t + 1 < d) v.y = x[t + 1];
            if (t + 2 < d) v.z = x[t + 2];
            if (t + 3 < d) v.w = x[t + 3];
        }
        x2 = fmaf(v.w, v.w, fmaf(v.z, v.z, fmaf(v.y, v.y, fmaf(v.x, v.x, x2))));
        xm2[t] = -2.0f * v.x;
        xm2[t + 1] = -2.0f * v.y;
        xm2[t + 2] = -2.0f * v.z;
        xm2[t + 3] = -2.0f * v.w;
    }
    float b1 = INFINITY, b2 = INFINITY;
    int bi = 0;
#pragma unroll 1
    for (int j0 = 0; j0 < k; j0 += 4) {            // kpad is a multiple of 128
        const float4 n4 = __ldg(reinterpret_cast<const float4*>(cnorm + j0));
        float a[4] = {n4.x, n4.y, n4.z, n4.w};
        const float* ct = c32t + j0;
#pragma unroll
        for (int t = 0; t < DP; ++t) {
            if (FULL || t < d) {
                const float4 w = __ldg(reinterpret_cast<const float4*>(ct + (long long)t * kpad));
                a[0] = fmaf(xm2[t], w.x, a[0]);
                a[1] = fmaf(xm2[t], w.y, a[1]);
                a[2] = fmaf(xm2[t], w.z, a[2]);
                a[3] = fmaf(xm2[t], w.w, a[3]);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float v = j0 + q < k ? a[q] : INFINITY;      // padding may hold anything
            b2 = fminf(b2, fmaxf(b1, v));
            if (v < b1) { b1 = v; bi = j0 + q; }
        }
    }
    return b2 - b1 > tie_kappa(d) * (thr_base + x2) + tie_abs(d + 1) ? bi : -1;
}

// Open rows of a 32-row unit from which decide_fp32_lanes is cheaper than as many
// decide_fp32_row: instructions of the one over those of the other.
__device__ __forceinline__ int lanes_from(int d, int k)
{
    return (k + 3) / 4 * (5 * d + 16) / ((k + 63) / 64 * 5 * d + 60) + 1;
}

}  // namespace km2
