// rt_newton.cuh -- the per-vertex temperature solve of the fixed point
// (Section 1.3, the balance of Eq. (RTb) discretised over the frequency grid):
// sum_nu wt_nu B_nu(T) = rhs with B_nu(T) = nu^3 / expm1(nu / T), to
// |dT| <= 1e-14 T in FP64.
//
// An FP64 operation costs 64 FP32 ones on this part, so the safeguarded Newton
// iteration (bisection bracket) runs in FP32 and one FP64 evaluation at its
// root finishes: Halley's step has a cubic error, which from an FP32 root
// (about 1e-7 off) is far below 1e-14.  Where that bound does not hold the
// FP64 Newton iteration goes on, and whenever FP32 cannot represent the problem
// the plain FP64 iteration runs from the previous T.  A step that is within
// the stopping rule ends the iteration before the bracket is looked at: a step
// that rounds to zero lies on a bracket end, and bisecting there threw the
// iterate back to the middle of the bracket.
// Bound: FP64 issue.  One temperature update on GB300 (before: three or more
// FP64 evaluations, each with an expm1 and four divisions a frequency):
// 41^3 x 64 channels 3.24 -> 0.55 ms, 32^3 x 16 0.96 -> 0.105 ms, 13^3 x 3 225 -> 14 us.
#pragma once

#include <cstdint>

namespace rt {

// LPV lanes per vertex (the power of two >= F, at most 32; 32 / LPV vertices
// per warp), lanes over the frequencies; the first two of a lane stay in
// registers.  With x = nu / T, r = 1 / expm1(x), B = nu^3 r:
//   T B' = B x (1 + r),  T B'' = B' (x (1 + 2 r) - 2).
// Sums over a vertex's lanes use shuffles masked to its LPV lanes, so the
// vertices of a warp iterate independently.
template <int LPV>
__device__ __forceinline__ unsigned seg_mask(int lane)
{
    if constexpr (LPV == 32) return 0xffffffffu;
    return ((1u << LPV) - 1u) << (lane & ~(LPV - 1));
}

template <int LPV>
struct LaneFreqs {
    const double* fq;
    int F, sl;
    double nu[2], c[2];   // nu and wt nu^3 (0 past the end)
    float nuf[2], cf[2];
    __device__ __forceinline__ LaneFreqs(const double* fq_, int F_, int lane) : fq(fq_), F(F_), sl(lane & (LPV - 1))
    {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int f = sl + k * LPV;
            nu[k] = f < F ? fq[4 * f] : 1.0;
            c[k] = f < F ? fq[4 * f + 1] * nu[k] * nu[k] * nu[k] : 0.0;
            nuf[k] = (float)nu[k];
            cf[k] = (float)c[k];
        }
    }
};

template <int LPV, class R>
__device__ __forceinline__ R lane_sum(R v, int lane)
{
    const unsigned m = seg_mask<LPV>(lane);
#pragma unroll
    for (int o = LPV >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(m, v, o);
    return v;
}

// g = sum wt B and dg = g' in FP64 (t > 0 or both zero)
template <int LPV>
__device__ __forceinline__ void planck64(const LaneFreqs<LPV>& L, double t, int lane, double& g, double& dg)
{
    g = dg = 0.0;
    if (t > 0.0) {
        const double it = 1.0 / t;
        auto add = [&](double nu, double c) {
            const double x = nu * it;
            if (x < 700.0) {
                const double r = 1.0 / expm1(x), B = c * r;
                g += B;
                dg += B * x * (1.0 + r);
            }
        };
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (L.c[k] != 0.0) add(L.nu[k], L.c[k]);
        for (int f = L.sl + 2 * LPV; f < L.F; f += LPV) {
            const double nu = L.fq[4 * f];
            add(nu, L.fq[4 * f + 1] * nu * nu * nu);
        }
        dg *= it;
    }
    g = lane_sum<LPV>(g, lane);
    dg = lane_sum<LPV>(dg, lane);
}

// the same in FP32, with q = g'' / g'
template <int LPV>
__device__ __forceinline__ void planck32(const LaneFreqs<LPV>& L, float t, int lane, float& g, float& dg, float& q)
{
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    const float it = 1.f / t;
    auto add = [&](float nu, float c) {
        const float x = nu * it;
        if (x < 80.f) {
            const float r = __fdividef(1.f, expm1f(x)), B = c * r, d = B * x * (1.f + r);
            s0 += B;
            s1 += d;
            s2 += d * (fmaf(2.f * x, r, x) - 2.f);
        }
    };
    if (t > 0.f) {
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (L.cf[k] != 0.f) add(L.nuf[k], L.cf[k]);
        for (int f = L.sl + 2 * LPV; f < L.F; f += LPV) {
            const float nu = (float)L.fq[4 * f];
            add(nu, (float)L.fq[4 * f + 1] * nu * nu * nu);
        }
    }
    g = lane_sum<LPV>(s0, lane);
    s1 = lane_sum<LPV>(s1, lane);
    s2 = lane_sum<LPV>(s2, lane);
    dg = s1 * it;
    q = s1 > 0.f ? s2 / s1 * it : 0.f;
}

// Safeguarded Newton for sum_nu wt_nu B_nu(T) = rhs in FP64, started from t in
// the bracket [lo, hi] (g(lo) <= rhs <= g(hi)); stops when a step moves T by at
// most 1e-14 T.  Returns false after 100 steps without that.
template <int LPV>
__device__ __noinline__ bool newton64(const double* __restrict__ fq, int F, double rhs, int lane, double& t, double lo, double hi)
{
    const LaneFreqs<LPV> L(fq, F, lane);
    double g, dg;
    for (int it = 0; it < 100; ++it) {
        planck64<LPV>(L, t, lane, g, dg);
        const double fv = g - rhs;
        if (fv < 0.0) lo = t;
        if (fv > 0.0) hi = t;
        double tn = dg > 0.0 ? t - fv / dg : 0.5 * (lo + hi);
        if (dg > 0.0 && fabs(tn - t) <= 1e-14 * fabs(tn)) {
            t = tn;
            return true;
        }
        if (!(tn > lo && tn < hi)) tn = 0.5 * (lo + hi);
        const bool done = fabs(tn - t) <= 1e-14 * fabs(tn);
        t = tn;
        if (done || fv == 0.0) return true;
    }
    return false;
}

// FP64 bracket [0, hi] by doubling from max(1, 2 tp), then Newton from tp
template <int LPV>
__device__ __noinline__ bool newton64_full(const double* __restrict__ fq, int F, double rhs, int lane, double tp, double& t)
{
    const LaneFreqs<LPV> L(fq, F, lane);
    double lo = 0.0, hi = fmax(1.0, 2.0 * tp);
    double g, dg;
    planck64<LPV>(L, hi, lane, g, dg);
    int guard = 0;
    while (g < rhs && guard < 200) {
        lo = hi;
        hi *= 2.0;
        planck64<LPV>(L, hi, lane, g, dg);
        ++guard;
    }
    t = (tp > lo && tp < hi) ? tp : 0.5 * (lo + hi);
    return newton64<LPV>(fq, F, rhs, lane, t, lo, hi);
}

// The same safeguarded Newton iteration in FP32: returns the FP32 root, the
// last bracket and q = g'' / g' there, or false when FP32 cannot represent the
// problem (rhs out of the normal range, no bracket, no convergence).
template <int LPV>
__device__ __forceinline__ bool newton32(const LaneFreqs<LPV>& L, double rhs, int lane, double tp, float& t, float& lo,
                                         float& hi, float& q)
{
    if (!(rhs > 1e-30 && rhs < 1e30)) return false;
    const float r = (float)rhs;
    float g, dg;
    lo = 0.f;
    hi = fmaxf(1.f, 2.f * (float)tp);
    planck32<LPV>(L, hi, lane, g, dg, q);
    int guard = 0;
    while (g < r && guard < 100) {
        lo = hi;
        hi *= 2.f;
        planck32<LPV>(L, hi, lane, g, dg, q);
        ++guard;
    }
    if (!(g >= r)) return false;
    const float tpf = (float)tp;
    t = (tpf > lo && tpf < hi) ? tpf : 0.5f * (lo + hi);
    for (int it = 0; it < 60; ++it) {
        planck32<LPV>(L, t, lane, g, dg, q);
        const float fv = g - r;
        if (fv < 0.f) lo = t;
        if (fv > 0.f) hi = t;
        float tn = dg > 0.f ? t - fv / dg : 0.5f * (lo + hi);
        if (dg > 0.f && fabsf(tn - t) <= 3e-6f * fabsf(tn)) {
            t = tn;
            return t > 0.f;
        }
        if (!(tn > lo && tn < hi)) tn = 0.5f * (lo + hi);
        const bool done = fabsf(tn - t) <= 3e-6f * fabsf(tn);
        t = tn;
        if (done || fv == 0.f) return t > 0.f;
    }
    return false;
}

// T for one vertex (LPV lanes, all of them call): false when no iteration met
// the stopping rule within its step limit
template <int LPV>
__device__ __forceinline__ bool solve_temperature(const double* __restrict__ fq, int F, double rhs, int lane, double tp, double& t)
{
    const LaneFreqs<LPV> L(fq, F, lane);
    float t32, lo32, hi32, q;
    bool ok = false;
    if (newton32<LPV>(L, rhs, lane, tp, t32, lo32, hi32, q)) {
        // Halley's step at the FP32 root; the next correction is about d (d q)^2
        double g, dg;
        t = (double)t32;
        planck64<LPV>(L, t, lane, g, dg);
        const double d = (g - rhs) / dg, z = d * (double)q;
        if (fabs(d) <= 1e-5 * t && fabs(d) * (z * z + 1e-10) <= 1e-15 * t) {
            t -= d / (1.0 - 0.5 * z);
            return true;
        }
        // polish in FP64 inside the FP32 bracket widened by 1e-4 (an FP32 sign
        // test can misjudge only points within FP32 rounding of the root)
        const double lo = (double)lo32 * (1.0 - 1e-4), hi = (double)hi32 * (1.0 + 1e-4);
        ok = newton64<LPV>(fq, F, rhs, lane, t, lo, hi);
        // a root pressed against a bracket end means the bracket was wrong
        if (ok && (fabs(t - lo) <= 1e-12 * t || fabs(t - hi) <= 1e-12 * t)) ok = false;
    }
    if (!ok) ok = newton64_full<LPV>(fq, F, rhs, lane, tp, t);
    return ok;
}

}  // namespace rt
