// rt_phase.cuh -- FP32 kernel values from tabulated phases (the hot evaluator
// of rows and columns of G).
//
// With A = 2 pi x and so on, 4 sinA sinB sinC = sin(f1) + sin(f2) - sin(f3) -
// sin(f4), f1 = C + (A - B), f2 = C - (A - B), f3 = C + (A + B), f4 = C - (A +
// B).  Along a straight segment from a to b every f_k is affine, so
//   mean of sin f_k = (cos f_k(a) - cos f_k(b)) / (f_k(b) - f_k(a)),
// and the four cosines belong to the end points: they are tabulated once per
// vertex and per quadrature point, and an optical depth costs four
// differences and one division (the four quotients share one reciprocal).  The
// Gauss rule of n >= 16 nodes gives the same number within 2e-14 for segments
// with |dx| + |dy| + |dz| <= 3 (rt_entry.cuh), which the box of the domain
// guarantees here.
//
// Reflected path x -> x' -> y on a wall normal to the axis of C, at C0: with Z
// = 2 C0 - C_x - C_y the rate of C is Z on the first leg and -Z on the second
// (per unit of the whole path), so the legs share the denominators Z + dv, Z -
// dv, Z + du, Z - du (du, dv = differences of A + B and A - B between x and y),
// and x' enters only through 2 cos C0 cos v' and 2 cos C0 cos u':
//   (c1x + c2y - hv)/(Z + dv) + (c2x + c1y - hv)/(Z - dv)
//     - (c3x + c4y - hu)/(Z + du) - (c4x + c3y - hu)/(Z - du).
// Coordinates are permuted so that the wall's axis comes last (p, q, c).
//
// A quotient whose denominator is small loses digits (numerator and
// denominator both carry FP32 rounding), so below kSmallDir / kSmallRefl turns
// it is replaced by sin(midpoint) times the sinc series, the form that
// gauss_sum_sinprod (rt_entry.cuh) evaluates everywhere.
#pragma once

#include "rt_entry.cuh"

namespace rt {

constexpr float kSmallDir = 1.f / 32.f;    // turns: table cosines are good to 3e-8
constexpr float kSmallRefl = 1.f / 16.f;   // turns: cos u', cos v' come from the SFU, 4e-7
constexpr float kTetB = 0.1381966011250105f;           // 4-point rule: weight of the other vertices
constexpr float kTetG = 0.5854101966249685f - kTetB;   // and what the point's own vertex has more

__device__ __forceinline__ float ex2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_approx(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// exp(-c tau) with -c log2(e) = hi + lo, the exponent rounded once.  ex2.approx
// rounds down: measured on GB300 its mean relative error is -4.9e-8 for results
// over a binade and -2.3e-8 for results in [0.87, 1], and the repeated products
// below would add that up (2.0e-7 in a matvec against 1.3e-7 without the bias).
// The exponent is raised by the same amount.
constexpr float kExpBias = 7.0e-8f;       // 4.9e-8 log2(e)
constexpr float kStepBias = 3.5e-8f;      // for exp(-dc tau), near 1
__device__ __forceinline__ float group_exp(float hi, float lo, float tau, float bias = kExpBias)
{
    return ex2_approx(fmaf(hi, tau, fmaf(lo, tau, bias)));
}

// a finished sum times c_g.  c_g has a remainder as in the exponent: rounding it
// here alone would shift every entry of the group one way (up to 6e-8).
__device__ __forceinline__ float times_c(const KernelParams& P, float v, int g) { return fmaf(v, P.cf[g], v * P.cflo[g]); }

// pairs of FP32 values in one 64-bit register: one instruction for two groups
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Sums over a chunk of MG groups (g0 .. g0 + MG - 1): e_g += w exp(-c_g tau).
// Slots beyond the last group hold values that nothing reads.
template <int MG>
struct GroupSum {
    static_assert(MG % 4 == 0, "groups come in float4 stores");
    f32x2 e[MG / 2];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int h = 0; h < MG / 2; ++h) e[h] = 0ull;
    }
    __device__ __forceinline__ void add(const KernelParams& P, int g0, float w, float tau)
    {
        if (P.c_arith) {
            // exp(-c_{g0+g} tau) = exp(-c_{g0} tau) exp(-dc tau)^g, two groups a step;
            // a fresh exponential every eight groups keeps the products' rounding short
            const float D = group_exp(P.dcl, P.dclo, tau, kStepBias);
            const float DD = D * D;
            const f32x2 d2 = pack2(DD, DD);
#pragma unroll
            for (int b = 0; b < MG; b += 8) {
                const float E = w * group_exp(P.cl[g0 + b], P.clo[g0 + b], tau);
                f32x2 p = pack2(E, E * D);
#pragma unroll
                for (int h = b / 2; h < (b + 8 < MG ? b + 8 : MG) / 2; ++h) {
                    e[h] = add2(e[h], p);
                    p = mul2(p, d2);
                }
            }
        } else {
#pragma unroll
            for (int h = 0; h < MG / 2; ++h)
                e[h] = add2(e[h], pack2(w * group_exp(P.cl[g0 + 2 * h], P.clo[g0 + 2 * h], tau),
                                        w * group_exp(P.cl[g0 + 2 * h + 1], P.clo[g0 + 2 * h + 1], tau)));
        }
    }
    __device__ __forceinline__ void add(const GroupSum& o)
    {
#pragma unroll
        for (int h = 0; h < MG / 2; ++h) e[h] = add2(e[h], o.e[h]);
    }
    __device__ __forceinline__ void store(float* row) const
    {
        float4* d = reinterpret_cast<float4*>(row);
#pragma unroll
        for (int k = 0; k < MG / 4; ++k) {
            float4 v;
            unpack2(e[2 * k], v.x, v.y);
            unpack2(e[2 * k + 1], v.z, v.w);
            d[k] = v;
        }
    }
    // row <- b this + g row
    __device__ __forceinline__ void blend(float* row, float b, float g) const
    {
        float4* d = reinterpret_cast<float4*>(row);
        const f32x2 bb = pack2(b, b), gg = pack2(g, g);
#pragma unroll
        for (int k = 0; k < MG / 4; ++k) {
            float4 v = d[k];
            const f32x2 lo = fma2(bb, e[2 * k], mul2(gg, pack2(v.x, v.y)));
            const f32x2 hi = fma2(bb, e[2 * k + 1], mul2(gg, pack2(v.z, v.w)));
            unpack2(lo, v.x, v.y);
            unpack2(hi, v.z, v.w);
            d[k] = v;
        }
    }
    // row += b this
    __device__ __forceinline__ void add_to(float* row, float b) const
    {
        float4* d = reinterpret_cast<float4*>(row);
        const f32x2 bb = pack2(b, b);
#pragma unroll
        for (int k = 0; k < MG / 4; ++k) {
            float4 v = d[k];
            const f32x2 lo = fma2(bb, e[2 * k], pack2(v.x, v.y));
            const f32x2 hi = fma2(bb, e[2 * k + 1], pack2(v.z, v.w));
            unpack2(lo, v.x, v.y);
            unpack2(hi, v.z, v.w);
            d[k] = v;
        }
    }
    __device__ __forceinline__ float get(int g) const
    {
        float a = 0.f, b = 0.f, r = 0.f;
#pragma unroll
        for (int h = 0; h < MG / 2; ++h) {
            unpack2(e[h], a, b);
            r = g == 2 * h ? a : (g == 2 * h + 1 ? b : r);
        }
        return r;
    }
};

template <>
struct GroupSum<1> {
    float e;
    __device__ __forceinline__ void zero() { e = 0.f; }
    __device__ __forceinline__ void add(const KernelParams& P, int g0, float w, float tau)
    {
        e = fmaf(w, group_exp(P.cl[g0], P.clo[g0], tau), e);
    }
    __device__ __forceinline__ void add(const GroupSum& o) { e += o.e; }
    __device__ __forceinline__ void store(float* row) const { row[0] = e; }
    __device__ __forceinline__ void blend(float* row, float b, float g) const { row[0] = fmaf(b, e, g * row[0]); }
    __device__ __forceinline__ void add_to(float* row, float b) const { row[0] = fmaf(b, e, row[0]); }
    __device__ __forceinline__ float get(int) const { return e; }
};

// A row's point x in permuted coordinates with its phases' cosines.
struct PhasePoint {
    float p, q, c, u, v;
    float4 cs;
};
__device__ __forceinline__ PhasePoint phase_point(const KernelParams& P, int i)
{
    const float4 a = P.pxyz[i];
    return {a.x, a.y, a.z, a.x + a.y, a.x - a.y, P.pcos[i]};
}

// n1/d1 + n2/d2 - n3/d3 - n4/d4 over one reciprocal (every |d| >= 1/32)
__device__ __forceinline__ float four_quotients(const float (&n)[4], const float (&d)[4])
{
    const float a = fmaf(n[0], d[1], n[1] * d[0]);
    const float b = fmaf(n[2], d[3], n[3] * d[2]);
    const float da = d[0] * d[1], db = d[2] * d[3];
    return fmaf(a, db, -b * da) * rcp_approx(da * db);
}
// sin(pi s) / (pi s) for |s| <= 1/16 (truncation below 6e-9)
__device__ __forceinline__ float sinc_small(float s)
{
    const float ps = (float)kPi * s;
    const float p2 = ps * ps;
    return fmaf(p2, fmaf(p2, 1.f / 120.f, -1.f / 6.f), 1.f);
}
__device__ __forceinline__ float min_abs(const float (&d)[4])
{
    return fminf(fminf(fabsf(d[0]), fabsf(d[1])), fminf(fabsf(d[2]), fabsf(d[3])));
}

// Direct term from x to the point y: y4 = (p, q, c, weight), yc = its cosines.
// Returns the weight over r^2 and tau.
__device__ __forceinline__ void phase_direct(const KernelParams& P, const PhasePoint& x, const float4& y4, const float4& yc,
                                             float& w, float& tau)
{
    const float dp = y4.x - x.p, dq = y4.y - x.q, dc = y4.z - x.c;
    const float r2 = fmaf(dc, dc, fmaf(dq, dq, dp * dp));
    const float rs = rsqrt_approx(r2);
    float k = P.k0f;
    if (P.sinprod) {
        const float dv = dp - dq, du = dp + dq;
        float d[4] = {dc + dv, dc - dv, dc + du, dc - du};
        float n[4] = {x.cs.x - yc.x, x.cs.y - yc.y, x.cs.z - yc.z, x.cs.w - yc.w};
        if (min_abs(d) < kSmallDir) {
            const float f[4] = {x.c + x.v, x.c - x.v, x.c + x.u, x.c - x.u};
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if (fabsf(d[m]) < kSmallDir) {
                    n[m] = (float)(2.0 * kPi) * sin2pi_sfu(fmaf(0.5f, d[m], f[m])) * sinc_small(d[m]);
                    d[m] = 1.f;
                }
        }
        k = fmaf(P.amp8pi, four_quotients(n, d), k);
    }
    w = y4.w * rcp_approx(r2);
    tau = r2 * rs * k;
}

// Term reflected on the first wall (normal to the axis of c).
__device__ __forceinline__ void phase_reflected(const KernelParams& P, const PhasePoint& x, const float4& y4,
                                                const float4& yc, float& w, float& tau)
{
    const float dp = y4.x - x.p, dq = y4.y - x.q, Z = P.wc0x2 - x.c - y4.z;
    const float r2 = fmaf(Z, Z, fmaf(dq, dq, dp * dp));
    const float rs = rsqrt_approx(r2);
    float k = P.k0f;
    if (P.sinprod) {
        const float dv = dp - dq, du = dp + dq;
        // x' splits the line from the image at t in [0, 1]; t = 0 where x and y lie in the
        // wall's plane or rounding puts y behind it (wall_point), which also keeps 0 / 0
        // out: a vertex on the wall sees a tetrahedron that is flat against it in FP32
        const float h = P.wc0 - x.c;
        const float t = h * Z > 0.f ? h * rcp_approx(Z) : 0.f;
        const float v1 = fmaf(t, dv, x.v), u1 = fmaf(t, du, x.u);
        const float hv = P.wcos2 * __cosf((float)(2.0 * kPi) * (v1 - rintf(v1)));
        const float hu = P.wcos2 * __cosf((float)(2.0 * kPi) * (u1 - rintf(u1)));
        float d[4] = {Z + dv, Z - dv, Z + du, Z - du};
        float n[4] = {x.cs.x + yc.y - hv, x.cs.y + yc.x - hv, x.cs.z + yc.w - hu, x.cs.w + yc.z - hu};
        if (min_abs(d) < kSmallRefl) {
            const float s = 1.f - t;
            // phases at x' as f1 (or f3) and f2 (or f4); the quotient over Z + dv is
            // leg 1 of f1 and leg 2 of f2, over Z - dv leg 1 of f2 and leg 2 of f1
            const float f[4] = {P.wc0 + v1, P.wc0 - v1, P.wc0 + u1, P.wc0 - u1};
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if (fabsf(d[m]) < kSmallRefl) {
                    const float a = t * d[m], b = s * d[m];
                    n[m] = (float)(2.0 * kPi) * (t * sin2pi_sfu(fmaf(-0.5f, a, f[m])) * sinc_small(a) +
                                                 s * sin2pi_sfu(fmaf(-0.5f, b, f[m ^ 1])) * sinc_small(b));
                    d[m] = 1.f;
                }
        }
        k = fmaf(P.amp8pi, four_quotients(n, d), k);
    }
    w = P.R0f * y4.w * rcp_approx(r2);
    tau = r2 * rs * k;
}

// ---- tables -------------------------------------------------------------------
// cosines of the four phases of a point (permuted coordinates); the arguments
// are reduced to half a turn in FP64, where the sums are exact
__device__ __forceinline__ float4 phase_cosines(float p, float q, float c)
{
    const double v = (double)p - (double)q, u = (double)p + (double)q;
    const double f[4] = {c + v, c - v, c + u, c - u};
    float r[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) r[k] = cospif(2.f * (float)(f[k] - rint(f[k])));
    return make_float4(r[0], r[1], r[2], r[3]);
}
__device__ __forceinline__ float axis_of(const Vec3<float>& a, int d) { return d == 0 ? a.x : (d == 1 ? a.y : a.z); }

// per vertex: permuted coordinates and cosines
static __global__ void phase_vertex_table(KernelParams P, float4* xyz, float4* cs)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.N) return;
    const Vec3<float> a = load_xyz<float>(P, i);
    const float p = axis_of(a, P.axis[0]), q = axis_of(a, P.axis[1]), c = axis_of(a, P.axis[2]);
    xyz[i] = make_float4(p, q, c, 0.f);
    cs[i] = phase_cosines(p, q, c);
}

// per tetrahedron: centroid and squared near limit; per point of the 4-point
// rule: coordinates and |T| w kappa(y) / 4 pi, and (phase evaluator) cosines
template <bool PHASE, bool XT>
__global__ void tet_point_table(KernelParams P, float4* cen4, float4* pts, float4* cs)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= P.T) return;
    const int4 tv = P.tet[t];
    const Vec3<float> v0 = load_xyz<float>(P, tv.x), v1 = load_xyz<float>(P, tv.y), v2 = load_xyz<float>(P, tv.z),
                      v3 = load_xyz<float>(P, tv.w);
    Vec3<float> cen;
    float diam, vol;
    load_tgeo<float>(P, t, cen, diam, vol);
    cen4[t] = make_float4(cen.x, cen.y, cen.z, 4.f * diam * diam);
    const float inv4pi = (float)(1.0 / (4.0 * kPi));
    for (int q = 0; q < 4; ++q) {
        const float b0 = tet_b<float>(q, 0), b1 = tet_b<float>(q, 1), b2 = tet_b<float>(q, 2), b3 = tet_b<float>(q, 3);
        const Vec3<float> y = {b0 * v0.x + b1 * v1.x + b2 * v2.x + b3 * v3.x, b0 * v0.y + b1 * v1.y + b2 * v2.y + b3 * v3.y,
                               b0 * v0.z + b1 * v1.z + b2 * v2.z + b3 * v3.z};
        const float w = vol * tet_w<float>(q) * inv4pi;
        if constexpr (PHASE) {
            float kap = P.k0f;
            if (P.sinprod) kap = fmaf(P.ampf, sinpif(2.f * y.x) * sinpif(2.f * y.y) * sinpif(2.f * y.z), kap);
            const float p = axis_of(y, P.axis[0]), qq = axis_of(y, P.axis[1]), c = axis_of(y, P.axis[2]);
            pts[(int64_t)q * P.T + t] = make_float4(p, qq, c, w * kap);
            if (P.sinprod) cs[(int64_t)q * P.T + t] = phase_cosines(p, qq, c);
        } else {
            pts[(int64_t)q * P.T + t] = make_float4(y.x, y.y, y.z, w * kappa_at<float, XT>(P, y.x, y.y, y.z));
        }
    }
}

}  // namespace rt
