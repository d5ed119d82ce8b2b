// screen.cuh -- the FP32 distance screen and its FP64 recheck, shared by the BCCP kernels (wspd.cu)
// and the nearest-component search (boruvka.cu).
#pragma once

#include "wspd.cuh"

namespace wm {

namespace {

// threshold of the FP32 screen: any candidate whose screened value exceeds T cannot beat the
// screened minimum s once both are evaluated exactly in FP64.  With an exact FP32 copy (eta = 0)
// T = s (1 + 4 eps32) + 1.5e-42; otherwise the copy's distance error eta comes on top on both sides:
// T = (sqrt(s (1 + 2 eps32)) + 2 eta)^2 (1 + 4 eps32) + 1.5e-42 (the second factor also covers the
// 2^-46 of the FP64 evaluations).  Both are bounded from above in FP32 with directed rounding (a
// float >= the exact value is >= its rounded-up value too): the FP64 pipe, where two square roots
// would cost more than the pass that asks for them, is not touched.
__device__ inline float screen_threshold(float s, const TravArgs &a)
{
    if (a.exact32) return __fadd_ru(__fmul_ru(s, 1.0f + 4.0f / 524288.0f), 1.6e-42f);
    const float q = __fadd_ru(__fsqrt_ru(__fmul_ru(s, 1.0f + 2.0f / 524288.0f)), a.eta2_f);
    return __fadd_ru(__fmul_ru(__fmul_ru(q, q), 1.0f + 4.0f / 524288.0f), 1.6e-42f);
}

// True when a screened value s proves that the exact FP64 weight of its point pair is at or above
// rho_hi, so that the pair's edge cannot belong to this round and needs no FP64 recheck: s is at
// least TravArgs::above_f, the smallest float whose rigorous lower bound on that weight reaches
// rho_hi (computed on the host, see above_threshold).
__device__ inline bool screened_above(float s, const TravArgs &a) { return s >= a.above_f; }

__device__ inline float dist32(const float *__restrict__ x32, int n, int d, int i, int j)
{
    float s = 0.f;
    for (int k = 0; k < d; ++k) {
        float t = x32[(size_t)k * n + i] - x32[(size_t)k * n + j];
        s = fmaf(t, t, s);
    }
    return s;
}

// dist32 with the dimension fixed at compile time (D > 0), the same operations in the same order
template <int D>
__device__ inline float dist32t(const float *__restrict__ x32, int n, int d, int i, int j)
{
    if (D <= 0) return dist32(x32, n, d, i, j);
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < (D > 0 ? D : 1); ++k) {
        float t = x32[(size_t)k * n + i] - x32[(size_t)k * n + j];
        s = fmaf(t, t, s);
    }
    return s;
}

// dist32 from the point-major copy: the same subtractions and fused multiply-adds in dimension
// order (a padded coordinate is 0 on both sides and adds exactly 0)
template <int D>
__device__ inline float dist32p(const float4 *__restrict__ x4, int i, int j)
{
    constexpr int Q = (D + 3) / 4;                          // float4s holding coordinates
    constexpr int S = Q <= 1 ? 1 : Q <= 2 ? 2 : 4;          // float4s per point (dp / 4)
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < Q; ++c) {
        const float4 p = x4[(size_t)i * S + c];
        const float4 q = x4[(size_t)j * S + c];
        const float pv[4] = {p.x, p.y, p.z, p.w}, qv[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (4 * c + r < D) {
                const float t = pv[r] - qv[r];
                s = fmaf(t, t, s);
            }
        }
    }
    return s;
}

__device__ inline double dist64(const double *__restrict__ x64, int n, int d, int i, int j)
{
    double s = 0.0;
    for (int k = 0; k < d; ++k) {
        double t = __dsub_rn(x64[(size_t)k * n + i], x64[(size_t)k * n + j]);
        s = __dadd_rn(s, __dmul_rn(t, t));
    }
    return s;
}

// max of two non-negative doubles through their bit patterns (integer compare, no FP64 op)
__device__ inline double pos_dmax(double x, double y)
{
    return __double_as_longlong(x) >= __double_as_longlong(y) ? x : y;
}

// True when the FP32 squared distance d32 of exact rows proves D <= cd2 for a core distance whose FP32 copy
// is c.  d32 is within 2^-19 of D and c within 2^-24 of cd2, and each besides within kAbsTiny (2^-140), which
// bounds what subnormal rounding takes: up to 2^-150 for each of 16 products, so that d32 can be 0 where D is
// above a cd2 that FP32 still holds.
__device__ inline bool proven_within(float d32, float c)
{
    return __fmaf_ru(d32, 1.0f + 1.0f / 131072.0f, 2.f * kAbsTiny) < __fmul_rd(c, 1.0f - 1.0f / 4194304.0f);
}

// exact FP64 weight of positions (i,j).  d32: the FP32 squared distance alone; c32: the larger
// FP32 core distance (HDBSCAN*).  When the distance is provably within the larger core distance, the
// weight is that core distance and the FP64 distance is skipped.
__device__ inline double exact_w2(const TravArgs &a, int i, int j, float d32, float c32)
{
    if (a.cd64) {
        double c = pos_dmax(a.cd64[i], a.cd64[j]);
        if (a.exact32 && proven_within(d32, c32)) return c;
        return pos_dmax(c, dist64(a.x64, a.n, a.d, i, j));
    }
    return dist64(a.x64, a.n, a.d, i, j);
}

// exact_w2, also noting the relative error of the FP32 screened value (sd, or for HDBSCAN* its
// maximum with the FP32 core distances c32) against the exact weight in err
__device__ inline double checked_w2(const TravArgs &a, int i, int j, float sd, float c32, float &err)
{
    const double w = exact_w2(a, i, j, sd, c32);
    if (w > 0.0) {   // the ratio in FP32 with outward rounding (a single FP64 subtraction)
        const double sv = a.cd64 ? pos_dmax((double)sd, (double)c32) : (double)sd;
        err = fmaxf(err, __fdiv_ru(__double2float_ru(fabs(sv - w)), __double2float_rd(w)));
    }
    return w;
}

// the largest relative screen error of a warp into stat[12] (bits of a non-negative float)
__device__ inline void err_flush(const TravArgs &a, float err)
{
    for (int o = 16; o; o >>= 1) err = fmaxf(err, __shfl_xor_sync(0xffffffffu, err, o));
    if ((threadIdx.x & 31) == 0 && err > 0.f) atomicMax(a.stat + 12, (unsigned long long)__float_as_uint(err));
}

// a recheck candidate held back so that the FP64 work of several lanes runs in one instruction
struct Deferred {
    int i = -1, j = 0;
    float sd = 0.f, c32 = 0.f;
};

__device__ inline float screen_value(const Deferred &c, bool hdb) { return hdb ? fmaxf(c.sd, c.c32) : c.sd; }

struct KMin {
    unsigned long long hi, lo;   // w2 bits, (min id << 32) | max id
};
__device__ inline void kmin_update(KMin &m, double w2, int pu, int pv)
{
    unsigned long long h = (unsigned long long)__double_as_longlong(w2);
    unsigned a = (unsigned)min(pu, pv), b = (unsigned)max(pu, pv);
    unsigned long long l = ((unsigned long long)a << 32) | b;
    if (h < m.hi || (h == m.hi && l < m.lo)) { m.hi = h; m.lo = l; }
}

__device__ inline unsigned long long warp_sum_u64(unsigned long long v)
{
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace

}  // namespace wm
