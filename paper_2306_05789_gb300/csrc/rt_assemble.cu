// rt_assemble.cu -- assembly of the operator on the GPU (Section 2, 2.1):
//   * constants: Gauss-Legendre nodes, tetrahedron and triangle rules
//   * entry kernels (warp per entry) for dense mode and arbitrary entry lists
//     (rows and columns of the H-matrix build: rt_rows.cuh)
//   * the emitter source Sbar^E
//   * batched partially pivoted ACA with pivots shared by all kappa groups
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <numeric>
#include <string>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "rt_entry.cuh"
#include "rt_internal.h"
#include "rt_pool.h"
#include "rt_rows.h"

namespace rt {


// ---------------------------------------------------------------------------
// host: quadrature tables
// ---------------------------------------------------------------------------
// Gauss-Legendre nodes: Newton iteration on P_n from the asymptotic guess
// cos(pi (4k + 3) / (4n + 2)); P_n and P_n' from the three-term recurrence.
void gauss_legendre_nodes(int n, std::vector<double>& t, std::vector<double>& w)
{
    t.assign(n, 0.0);
    w.assign(n, 0.0);
    for (int k = 0; k < n; ++k) {
        double x = std::cos(kPi * (4.0 * k + 3.0) / (4.0 * n + 2.0));
        double dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double pm = 1.0, p = x;
            for (int l = 1; l < n; ++l) {
                double pn = ((2.0 * l + 1.0) * x * p - l * pm) / (l + 1.0);
                pm = p;
                p = pn;
            }
            dp = n * (pm - x * p) / (1.0 - x * x);
            double step = p / dp;
            x -= step;
            if (std::fabs(step) <= 1e-16 * std::fabs(x) + 1e-300) break;
        }
        {
            double pm = 1.0, p = x;
            for (int l = 1; l < n; ++l) {
                double pn = ((2.0 * l + 1.0) * x * p - l * pm) / (l + 1.0);
                pm = p;
                p = pn;
            }
            dp = n * (pm - x * p) / (1.0 - x * x);
        }
        t[k] = x;
        w[k] = 2.0 / ((1.0 - x * x) * dp * dp);
    }
}

// Tetrahedron rules in barycentric coordinates: the symmetric 4-point rule of
// degree 2 and the positive 14-point rule of degree 5 (two S31 orbits, one S22
// orbit); triangle rules: 3-point degree 2 and Radon's 7-point degree 5.
static void tet_rules(double* b, double* w)
{
    const double al = (5.0 + 3.0 * std::sqrt(5.0)) / 20.0, be = (5.0 - std::sqrt(5.0)) / 20.0;
    int r = 0;
    for (int k = 0; k < 4; ++k, ++r) {
        for (int d = 0; d < 4; ++d) b[4 * r + d] = d == k ? al : be;
        w[r] = 0.25;
    }
    const double s31[2][2] = {{0.0927352503108912, 0.07349304311636196}, {0.3108859192633006, 0.1126879257180159}};
    for (int o = 0; o < 2; ++o)
        for (int k = 0; k < 4; ++k, ++r) {
            for (int d = 0; d < 4; ++d) b[4 * r + d] = d == k ? 1.0 - 3.0 * s31[o][0] : s31[o][0];
            w[r] = s31[o][1];
        }
    const double s22 = 0.4544962958743504, ws22 = 0.04254602077708147;
    for (int a = 0; a < 4; ++a)
        for (int c = a + 1; c < 4; ++c, ++r) {
            for (int d = 0; d < 4; ++d) b[4 * r + d] = (d == a || d == c) ? s22 : 0.5 - s22;
            w[r] = ws22;
        }
}

static void tri_rules(double* b, double* w)
{
    int r = 0;
    for (int k = 0; k < 3; ++k, ++r) {
        for (int d = 0; d < 3; ++d) b[3 * r + d] = d == k ? 2.0 / 3.0 : 1.0 / 6.0;
        w[r] = 1.0 / 3.0;
    }
    b[3 * r] = b[3 * r + 1] = b[3 * r + 2] = 1.0 / 3.0;
    w[r++] = 0.225;
    const double q = std::sqrt(15.0);
    const double orb[2][2] = {{(6.0 - q) / 21.0, (155.0 - q) / 1200.0}, {(6.0 + q) / 21.0, (155.0 + q) / 1200.0}};
    for (int o = 0; o < 2; ++o)
        for (int k = 0; k < 3; ++k, ++r) {
            for (int d = 0; d < 3; ++d) b[3 * r + d] = d == k ? 1.0 - 2.0 * orb[o][0] : orb[o][0];
            w[r] = orb[o][1];
        }
}

void quadrature_rules(double (&tet_b)[72], double (&tet_w)[18], double (&tri_b)[30], double (&tri_w)[10])
{
    tet_rules(tet_b, tet_w);
    tri_rules(tri_b, tri_w);
}

int assemble_setup_constants(Operator& op, std::string& err)
{
    std::vector<double> t, w;
    gauss_legendre_nodes(op.ngauss, t, w);
    for (int g = 0; g < kMaxGauss; ++g) {
        const double u = g < op.ngauss ? 0.5 * (1.0 + t[g]) : 0.0, hw = g < op.ngauss ? 0.5 * w[g] : 0.0;
        op.kp.gu64[g] = u;
        op.kp.gw64[g] = hw;
        op.kp.gu32[g] = (float)u;
        op.kp.gw32[g] = (float)hw;
    }
    // every unit at the first build, whichever of them it needs: the uploads wait for the
    // device, which a later build must not do while another thread captures a solve
    int rc;
    if ((rc = upload_rules(err))) return rc;
    if ((rc = RowEval<EV_PHASE>::setup(err))) return rc;
    if ((rc = RowEval<EV_PLAIN>::setup(err))) return rc;
    return RowEval<EV_GENERAL>::setup(err);
}

// ---------------------------------------------------------------------------
// entry kernels
// ---------------------------------------------------------------------------
constexpr int kWarpsPerCta = 8;

// Arbitrary (row, col) pairs, internal vertex ids.
template <class R, int MG, bool XT = false>
__global__ void __launch_bounds__(32 * kWarpsPerCta) entries_pairs_kernel(KernelParams P, int group, int64_t count,
                                                                          const int32_t* rows, const int32_t* cols,
                                                                          const int* iperm, double* out)
{
    __shared__ int s_tet[kWarpsPerCta][32], s_cnt[kWarpsPerCta][32], s_pre[kWarpsPerCta][33];
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * kWarpsPerCta;
    for (int64_t e = (int64_t)blockIdx.x * kWarpsPerCta + wib; e < count; e += nw) {
        int i = rows[e], j = cols[e];
        if (iperm) {
            i = iperm[i];
            j = iperm[j];
        }
        R acc[MG];
        entry_warp<R, MG, XT>(P, i, j, acc, s_tet[wib], s_cnt[wib], s_pre[wib]);
        R v = R(0);
#pragma unroll
        for (int g = 0; g < MG; ++g)
            if (g == group) v = acc[g];
        if (lane == 0) out[e] = (double)v;
    }
}

static int grid_for(int64_t warps)
{
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t ctas = (warps + kWarpsPerCta - 1) / kWarpsPerCta;
    int64_t cap = (int64_t)sms * 16;
    return (int)std::max<int64_t>(1, std::min(ctas, cap));
}

// Dispatch on the group count: the accumulator array is sized at compile time.
// general kernels (XT: further walls and corner terms, a kappa grid, opaque
// boxes): 16 or 64 group slots
#define RT_DISPATCH_MG_XT(G, MACRO) \
    do {                            \
        if ((G) <= 16) {            \
            MACRO(16, true);        \
        } else {                    \
            MACRO(64, true);        \
        }                           \
    } while (0)

#define RT_DISPATCH_MG(G, MACRO) \
    do {                         \
        if ((G) <= 1) {          \
            MACRO(1);            \
        } else if ((G) <= 4) {   \
            MACRO(4);            \
        } else if ((G) <= 8) {   \
            MACRO(8);            \
        } else if ((G) <= 16) {  \
            MACRO(16);           \
        } else if ((G) <= 32) {  \
            MACRO(32);           \
        } else {                 \
            MACRO(64);           \
        }                        \
    } while (0)

// ---------------------------------------------------------------------------
// dense mode: the whole matrix [G][N][N] row-major
// ---------------------------------------------------------------------------
// A sum of many terms: FP32 compensated (Kahan), FP64 plain.  A sum that has
// overflowed stays infinite: its compensation would be inf - inf.
template <class R>
struct Sum {
    R v = R(0), lost = R(0);
    __device__ __forceinline__ void add(R x)
    {
        if constexpr (sizeof(R) == 4) {
            const R y = x - lost, t = v + y;
            lost = isinf(t) ? R(0) : (t - v) - y;
            v = t;
        } else {
            v += x;
        }
    }
};

// A thread takes one tetrahedron of one row and evaluates every point once for
// the four hat functions of its vertices (entry by entry, each point was
// evaluated four times); the vertex sums go to scratch [row][vertex slot][g][T]
// and dense_gather adds each column's in the order of its tetrahedra.
// Bound: FP64 issue (1/64 of the FP32 rate): for a constant kappa a term is one
// rsqrt (1/r^2 and r; the broken path is as long as the line from the image when
// the mesh lies inside the wall) and one exponential.  12^3, kappa = 1, one wall,
// 1.2e8 terms: the whole matrix 117 ms entry by entry, 15.3 ms this way.
// Accuracy: the entry evaluator spreads an entry's points over 32 lanes, so the sums
// here are split too (FP64: per term, and a column's tetrahedra over eight) or
// compensated (FP32).  Root mean square error of an entry against extended precision,
// 5^3, oblique wall: FP64 2.03e-16 (entry evaluator 2.03e-16, serial sums 2.20e-16),
// FP32 1.17e-7 (1.16e-7; serial sums, rsqrt and one weight a point 1.40e-7).
constexpr int kDenseThreads = 128;
template <class R, int MG, bool XT>
__global__ void __launch_bounds__(kDenseThreads) dense_tets_kernel(KernelParams P, int row0, int g0, R* __restrict__ scratch)
{
    // FP64 sums every term of up to four groups by itself (registers for more would spill)
    constexpr bool by_term = sizeof(R) == 8 && MG <= 4;
    const int tet = blockIdx.x * kDenseThreads + threadIdx.x;
    if (tet >= P.T) return;
    const Vec3<R> xi = load_xyz<R>(P, row0 + blockIdx.y);
    Vec3<R> xb = xi;
    if (P.has_wall) xb = mirror_point<R>(P, xi);
    const int4 tv = P.tet[tet];
    const Vec3<R> v[4] = {load_xyz<R>(P, tv.x), load_xyz<R>(P, tv.y), load_xyz<R>(P, tv.z), load_xyz<R>(P, tv.w)};
    Vec3<R> cen;
    R diam, vol;
    load_tgeo<R>(P, tet, cen, diam, vol);
    const R lim = R(4) * diam * diam, inv4pi = R(1.0 / (4.0 * kPi));
    Sum<R> acc[4][MG];
    const int nt = XT ? 2 + P.n_extra : 2;
    for (int t = 0; t < nt; ++t) {
        if (t == 1 && !P.has_wall) continue;
        Vec3<R> src;
        R scale;
        term_source<R>(P, t, xi, xb, src, scale);
        const bool near = dist2<R>(src, cen) < lim;
        const int q0 = near ? 4 : 0, nq = near ? 14 : 4;
        Sum<R> part[by_term ? 4 : 1][MG];
        for (int q = q0; q < q0 + nq; ++q) {
            const R b[4] = {tet_b<R>(q, 0), tet_b<R>(q, 1), tet_b<R>(q, 2), tet_b<R>(q, 3)};
            const Vec3<R> y = {b[0] * v[0].x + b[1] * v[1].x + b[2] * v[2].x + b[3] * v[3].x,
                               b[0] * v[0].y + b[1] * v[1].y + b[2] * v[2].y + b[3] * v[3].y,
                               b[0] * v[0].z + b[1] * v[1].z + b[2] * v[2].z + b[3] * v[3].z};
            const R r2 = dist2<R>(src, y), kap = kappa_at<R, XT>(P, y.x, y.y, y.z);
            const bool straight = !XT && P.kappa_kind == RT_KAPPA_CONST && (t == 0 || P.wall_inside);
            R w[4], tau;
            if (!straight) {
                if constexpr (XT) {
                    tau = term_depth<R>(P, t, xi, src, y);
                    if (!(tau < R(INFINITY))) continue;   // path through an opaque box
                } else if (t == 0) {
                    tau = optical_depth<R>(P, xi, y);
                } else {
                    const Vec3<R> xp = wall_point<R>(P, src, y);
                    tau = optical_depth<R>(P, xi, xp) + optical_depth<R>(P, xp, y);
                }
            }
            if constexpr (sizeof(R) == 4) {
                // every hat function's weight as its own product and division: their
                // roundings differ from vertex to vertex and average out
                if (straight) tau = kp_k0<R>(P) * sqrt_r(r2);
#pragma unroll
                for (int k = 0; k < 4; ++k) w[k] = vol * tet_w<R>(q) * b[k] * kap * inv4pi / r2 * scale;
            } else {
                w[0] = scale * vol * tet_w<R>(q) * kap * inv4pi;
                if (straight) {
                    const R rs = rsqrt(r2);
                    tau = kp_k0<R>(P) * r2 * rs;
                    w[0] *= rs * rs;
                } else {
                    w[0] /= r2;
                }
            }
#pragma unroll
            for (int g = 0; g < MG; ++g)
                if (g0 + g < P.G) {
                    const R cg = kp_c<R>(P, g0 + g), E = exp_r(-cg * tau);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        Sum<R>& s = by_term ? part[by_term ? k : 0][g] : acc[k][g];
                        if constexpr (sizeof(R) == 4) s.add(w[k] * cg * E);
                        else s.v += b[k] * (w[0] * cg * E);
                    }
                }
        }
        if constexpr (by_term) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int g = 0; g < MG; ++g) acc[k][g].v += part[k][g].v;
        }
    }
    const int64_t row = (int64_t)blockIdx.y * 4 * MG;
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int g = 0; g < MG; ++g) scratch[(row + k * MG + g) * P.T + tet] = acc[k][g].v;
}

template <class R, int MG>
__global__ void __launch_bounds__(256) dense_gather(KernelParams P, int row0, int g0, const R* __restrict__ scratch, R* __restrict__ out)
{
    const int j = blockIdx.x * 256 + threadIdx.x;
    if (j >= P.N) return;
    const int t0 = P.vt_ptr[j], t1 = P.vt_ptr[j + 1];
    const int64_t row = (int64_t)blockIdx.y * 4 * MG;
    for (int g = 0; g < MG && g0 + g < P.G; ++g) {
        // eight partial sums, as the lanes of the entry evaluator keep them: one serial sum of
        // a column's 24 tetrahedra adds up more rounding than everything before it
        Sum<R> s[8];
        for (int e0 = t0; e0 < t1; e0 += 8)
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (e0 + k < t1) {
                    const int packed = P.vt_idx[e0 + k];
                    s[k].add(scratch[(row + (packed & 3) * MG + g) * P.T + (packed >> 2)]);
                }
        const R all = ((s[0].v + s[1].v) + (s[2].v + s[3].v)) + ((s[4].v + s[5].v) + (s[6].v + s[7].v));
        out[(int64_t)(g0 + g) * P.N * P.N + (int64_t)(row0 + blockIdx.y) * P.N + j] = all;
    }
}

template <class R, int MG>
static int dense_rows(Operator& op, R* out, cudaStream_t s, std::string& err)
{
    // rows at a time: 64 MB of vertex sums stay in L2 between the two kernels
    const int64_t per_row = (int64_t)4 * MG * op.T * sizeof(R);
    const int rows = (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(op.N, 32768), ((int64_t)64 << 20) / per_row));
    R* scratch = nullptr;
    if (cudaMallocAsync((void**)&scratch, (size_t)(rows * per_row), s) != cudaSuccess) {
        err = "cudaMallocAsync (dense assembly scratch) failed";
        return RT_ENOMEM;
    }
    for (int r0 = 0; r0 < op.N; r0 += rows) {
        const int nr = std::min(rows, op.N - r0);
        const dim3 ge((op.T + kDenseThreads - 1) / kDenseThreads, nr), gg((op.N + 255) / 256, nr);
        for (int g0 = 0; g0 < op.G; g0 += MG) {
            if (op.kp.ext) dense_tets_kernel<R, MG, true><<<ge, kDenseThreads, 0, s>>>(op.kp, r0, g0, scratch);
            else dense_tets_kernel<R, MG, false><<<ge, kDenseThreads, 0, s>>>(op.kp, r0, g0, scratch);
            dense_gather<R, MG><<<gg, 256, 0, s>>>(op.kp, r0, g0, scratch, out);
        }
    }
    cudaFreeAsync(scratch, s);
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
}

template <class R>
static int dense_matrix(Operator& op, cudaStream_t s, std::string& err)
{
    R* d = nullptr;
    int rc = dev_alloc(op, &d, (size_t)op.G * op.N * op.N, err);
    if (rc) return rc;
    op.d_dense = d;
    if (op.G <= 1) return dense_rows<R, 1>(op, d, s, err);
    if (op.G <= 4) return dense_rows<R, 4>(op, d, s, err);
    if (op.G <= 8) return dense_rows<R, 8>(op, d, s, err);   // 11^3, 8 groups: FP32 4.4 -> 2.7 ms, FP64 47 -> 41 ms
    return dense_rows<R, 16>(op, d, s, err);
}

int assemble_dense(Operator& op, cudaStream_t s, std::string& err)
{
    const int64_t N = op.N;
    const size_t esz = op.prec == RT_PREC_F64 ? 8 : 4;
    const int rc = op.prec == RT_PREC_F64 ? dense_matrix<double>(op, s, err) : dense_matrix<float>(op, s, err);
    if (rc) return rc;
    op.info.entries_evaluated += N * N;
    op.info.stored_entries = N * N;
    op.info.apply_bytes = (int64_t)op.F * N * N * (int64_t)esz + 2 * (int64_t)op.F * N * (int64_t)esz;
    op.info.apply_flops = 2 * (int64_t)op.F * N * N;
    return RT_OK;
}

int eval_entries(Operator& op, int group, int64_t count, const int32_t* rows, const int32_t* cols, double* out,
                 cudaStream_t s, std::string& err)
{
    if (count <= 0) return RT_OK;
    int grid = grid_for(count);
    const int* ip = op.d_iperm;
    if (op.prec == RT_PREC_F64) {
#define RT_LAUNCH_PAIRS(MG, XT) \
    entries_pairs_kernel<double, MG, XT><<<grid, 32 * kWarpsPerCta, 0, s>>>(op.kp, group, count, rows, cols, ip, out)
#define RT_LAUNCH_PAIRS1(MG) RT_LAUNCH_PAIRS(MG, false)
        if (op.kp.ext) RT_DISPATCH_MG_XT(op.G, RT_LAUNCH_PAIRS);
        else RT_DISPATCH_MG(op.G, RT_LAUNCH_PAIRS1);
#undef RT_LAUNCH_PAIRS1
#undef RT_LAUNCH_PAIRS
    } else {
#define RT_LAUNCH_PAIRS(MG, XT) \
    entries_pairs_kernel<float, MG, XT><<<grid, 32 * kWarpsPerCta, 0, s>>>(op.kp, group, count, rows, cols, ip, out)
#define RT_LAUNCH_PAIRS1(MG) RT_LAUNCH_PAIRS(MG, false)
        if (op.kp.ext) RT_DISPATCH_MG_XT(op.G, RT_LAUNCH_PAIRS);
        else RT_DISPATCH_MG(op.G, RT_LAUNCH_PAIRS1);
#undef RT_LAUNCH_PAIRS1
#undef RT_LAUNCH_PAIRS
    }
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
}

// ---------------------------------------------------------------------------
// emitter source Sbar^E (Example of Section 1.2, Section 2)
// ---------------------------------------------------------------------------
// Shat_g(x_i) = (1/4pi) int_{Gamma_Q} ([(x-y).n]_-)^2 e^{-c_g tau(x,y)}/|x-y|^4
//             + R0 ([(xbar-y).n]_-)^2 e^{-c_g(tau(x,x')+tau(x',y))}/|xbar-y|^4 dGamma(y),
// 7-point rule within two diameters of the triangle centroid, 3-point rule
// otherwise; a source point that is a vertex of the triangle contributes the
// limit (angle at the vertex)/(8 pi) (times R0 for the image term).
// One warp per vertex; lanes over triangles.  out[f][i] = Q_f Shat_{g(f)}(x_i).
template <class R, int MG>
__global__ void __launch_bounds__(256) source_kernel(KernelParams P, int n_emit, const int4* emit, const int* fgroup,
                                                     const double* Q, int F, R* out)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    const R inv4pi = R(1.0 / (4.0 * kPi));
    for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < P.N; i += nw) {
        const Vec3<R> xi = load_xyz<R>(P, (int)i);
        Vec3<R> xb = xi;
        bool on_wall = false;
        if (P.has_wall) {
            xb = mirror_point<R>(P, xi);
            on_wall = dist2<R>(xi, xb) <= R(1e-20);
        }
        R acc[MG];
#pragma unroll
        for (int g = 0; g < MG; ++g) acc[g] = R(0);
        for (int e = lane; e < n_emit; e += 32) {
            const int4 tv = emit[e];
            const Vec3<R> V0 = load_xyz<R>(P, tv.x), V1 = load_xyz<R>(P, tv.y), V2 = load_xyz<R>(P, tv.z);
            const Vec3<R> e1 = {V1.x - V0.x, V1.y - V0.y, V1.z - V0.z};
            const Vec3<R> e2 = {V2.x - V0.x, V2.y - V0.y, V2.z - V0.z};
            Vec3<R> nn = {e1.y * e2.z - e1.z * e2.y, e1.z * e2.x - e1.x * e2.z, e1.x * e2.y - e1.y * e2.x};
            const R a2 = sqrt_r(nn.x * nn.x + nn.y * nn.y + nn.z * nn.z);
            nn.x /= a2;
            nn.y /= a2;
            nn.z /= a2;
            const R area = R(0.5) * a2;
            const Vec3<R> cen = {(V0.x + V1.x + V2.x) / R(3), (V0.y + V1.y + V2.y) / R(3), (V0.z + V1.z + V2.z) / R(3)};
            R diam2 = dist2<R>(V0, V1);
            diam2 = fmax(diam2, dist2<R>(V0, V2));
            diam2 = fmax(diam2, dist2<R>(V1, V2));
            int vloc = tv.x == (int)i ? 0 : (tv.y == (int)i ? 1 : (tv.z == (int)i ? 2 : -1));
            for (int term = 0; term < 2 + P.n_extra; ++term) {
                if (term == 1 && !P.has_wall) continue;
                Vec3<R> src;
                R scale;
                term_source<R>(P, term, xi, xb, src, scale);
                // the source point is x itself: always for the direct term, for an
                // image when x lies on its wall(s)
                const bool at_x = term == 0 || (term == 1 ? on_wall : dist2<R>(xi, src) <= R(1e-20));
                if (vloc >= 0 && at_x) {
                    // limit at a vertex of the emitter: angle / (8 pi)
                    const Vec3<R> A = vloc == 0 ? V0 : (vloc == 1 ? V1 : V2);
                    const Vec3<R> B = vloc == 0 ? V1 : (vloc == 1 ? V2 : V0);
                    const Vec3<R> C = vloc == 0 ? V2 : (vloc == 1 ? V0 : V1);
                    const Vec3<R> u = {B.x - A.x, B.y - A.y, B.z - A.z}, v = {C.x - A.x, C.y - A.y, C.z - A.z};
                    R cs = (u.x * v.x + u.y * v.y + u.z * v.z) / sqrt_r((u.x * u.x + u.y * u.y + u.z * u.z) *
                                                                         (v.x * v.x + v.y * v.y + v.z * v.z));
                    cs = fmin(R(1), fmax(R(-1), cs));
                    const R lim = scale * acos(cs) * R(1.0 / (8.0 * kPi));
#pragma unroll
                    for (int g = 0; g < MG; ++g)
                        if (g < P.G) acc[g] += lim;
                    continue;
                }
                const R sd = (src.x - V0.x) * nn.x + (src.y - V0.y) * nn.y + (src.z - V0.z) * nn.z;
                if (!(sd < R(0))) continue;
                const R cm = -sd;
                const bool nearp = dist2<R>(src, cen) < R(4) * diam2;
                const int q0 = nearp ? 3 : 0, nq = nearp ? 7 : 3;
                for (int q = 0; q < nq; ++q) {
                    const R b0 = R(c_tri_b[3 * (q0 + q)]), b1 = R(c_tri_b[3 * (q0 + q) + 1]),
                            b2 = R(c_tri_b[3 * (q0 + q) + 2]);
                    const Vec3<R> y = {b0 * V0.x + b1 * V1.x + b2 * V2.x, b0 * V0.y + b1 * V1.y + b2 * V2.y,
                                       b0 * V0.z + b1 * V1.z + b2 * V2.z};
                    const R r2 = dist2<R>(src, y);
                    const R tau = term_depth<R>(P, term, xi, src, y);
                    const R geo = scale * area * R(c_tri_w[q0 + q]) * cm * cm / (r2 * r2) * inv4pi;
#pragma unroll
                    for (int g = 0; g < MG; ++g)
                        if (g < P.G) acc[g] += geo * exp_r(-kp_c<R>(P, g) * tau);
                }
            }
        }
#pragma unroll
        for (int g = 0; g < MG; ++g) {
            R v = acc[g];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            acc[g] = v;
        }
        if (lane == 0) {
            for (int f = 0; f < F; ++f) {
                R v = R(0);
#pragma unroll
                for (int g = 0; g < MG; ++g)
                    if (g == fgroup[f]) v = acc[g];
                out[(int64_t)f * P.N + i] = R(Q[f]) * v;
            }
        }
    }
}

int assemble_source(Operator& op, cudaStream_t s, std::string& err)
{
    int rc;
    int* d_fg = nullptr;
    double* d_Q = nullptr;
    RT_CUDA_TRY(cudaMallocAsync((void**)&d_fg, sizeof(int) * op.F, s));
    RT_CUDA_TRY(cudaMallocAsync((void**)&d_Q, sizeof(double) * op.F, s));
    RT_CUDA_TRY(cudaMemcpyAsync(d_fg, op.fgroup.data(), sizeof(int) * op.F, cudaMemcpyHostToDevice, s));
    RT_CUDA_TRY(cudaMemcpyAsync(d_Q, op.Q.data(), sizeof(double) * op.F, cudaMemcpyHostToDevice, s));
    const int grid = grid_for(op.N);
    if (op.vec64) {
        double* d = nullptr;
        if ((rc = dev_alloc(op, &d, (size_t)op.F * op.N, err))) return rc;
        op.d_SE = d;
#define RT_LAUNCH_SRC(MG) \
    source_kernel<double, MG><<<grid, 256, 0, s>>>(op.kp, op.n_emit, op.d_emit, d_fg, d_Q, op.F, d)
        RT_DISPATCH_MG(op.G, RT_LAUNCH_SRC);
#undef RT_LAUNCH_SRC
    } else {
        float* d = nullptr;
        if ((rc = dev_alloc(op, &d, (size_t)op.F * op.N, err))) return rc;
        op.d_SE = d;
#define RT_LAUNCH_SRC(MG) \
    source_kernel<float, MG><<<grid, 256, 0, s>>>(op.kp, op.n_emit, op.d_emit, d_fg, d_Q, op.F, d)
        RT_DISPATCH_MG(op.G, RT_LAUNCH_SRC);
#undef RT_LAUNCH_SRC
    }
    RT_CUDA_TRY(cudaGetLastError());
    RT_CUDA_TRY(cudaFreeAsync(d_fg, s));
    RT_CUDA_TRY(cudaFreeAsync(d_Q, s));
    return RT_OK;
}

void eval_tables_free(Operator& op)
{
    for (void* p : op.eval_tables) cudaFreeAsync(p, op.stream);
    op.eval_tables.clear();
    op.eval_bytes = 0;
    op.d_sub_tets = nullptr;
    op.d_subs = nullptr;
    op.d_pass_ref = nullptr;
    op.d_pass_run = nullptr;
    op.kp.pxyz = op.kp.pcos = op.kp.tcen = op.kp.tpt = op.kp.tcos = nullptr;
}

// a column cluster's sub-clusters: the nodes of at most kSubCols columns below it, in
// order; false where a leaf is wider
static bool sub_clusters(const Plan& P, int cluster, std::vector<int>& out)
{
    std::vector<int> stack = {cluster};
    while (!stack.empty()) {
        const int k = stack.back();
        stack.pop_back();
        const ClusterNode& C = P.clusters[k];
        if (C.size <= kSubCols) {
            out.push_back(k);
        } else if (C.left < 0) {
            return false;
        } else {
            stack.push_back(C.right);
            stack.push_back(C.left);
        }
    }
    return true;
}

static std::vector<char> column_clusters(const Plan& P)
{
    std::vector<char> used(P.clusters.size(), 0);
    for (const FarBlock& b : P.far_blocks) used[b.sc] = 1;
    for (const FarBlock& b : P.near_blocks) used[b.sc] = 1;
    return used;
}

int64_t eval_bytes_bound(const Plan& P, int64_t T, int G, int ev)
{
    const int mg = group_chunk(G, ev);
    const int64_t pt = (int64_t)tets_per_thread(mg, ev) * eval_threads(G, ev, P.far_blocks.size());
    int64_t bytes = T * (ev == EV_PHASE ? 144 : 80) + (ev == EV_PHASE ? (int64_t)P.N * 32 : 0);
    const std::vector<char> used = column_clusters(P);
    std::vector<char> seen(P.clusters.size(), 0);
    std::vector<int> sub;
    for (int c = 0; c < (int)P.clusters.size(); ++c) {
        if (!used[c]) continue;
        sub.clear();
        sub_clusters(P, c, sub);
        for (int k : sub) {
            if (seen[k]) continue;
            seen[k] = 1;
            const int64_t pairs = std::min<int64_t>(T, (int64_t)(4.0 * (double)T / P.N * P.clusters[k].size) + 1);
            const int64_t passes = (pairs + pt - 1) / pt;
            bytes += (int64_t)sizeof(SubInfo) + 4 * pairs + passes * (8 * pt + 4 * kRunWords + 4);
        }
    }
    for (const FarBlock& b : P.near_blocks) {
        const int rows = rows_per_item(mg, std::min(b.n, kSubCols));
        bytes += (int64_t)((b.m + rows - 1) / rows + 1) * (int64_t)sizeof(RowItem);
    }
    return bytes;
}

// sub-clusters of every column cluster and the tetrahedra touching each
int prepare_row_eval(Operator& op, std::string& err)
{
    const Plan& P = op.plan;
    const int nc = (int)P.clusters.size();
    op.sub_of_cluster_ptr.assign(nc + 1, 0);
    op.sub_of_cluster.clear();
    op.sub_start.clear();
    op.sub_size.clear();
    op.sub_tet_ptr.assign(1, 0);
    std::vector<int> sub_id(nc, -1), tets, stamp(op.T, -1);
    const std::vector<char> used = column_clusters(P);
    std::vector<std::vector<int>> subs(nc);
    for (int c = 0; c < nc; ++c)
        if (used[c] && !sub_clusters(P, c, subs[c])) {
            err = "cluster leaf larger than the row-evaluation width";
            return RT_EINVAL;
        }
    for (int c = 0; c < nc; ++c) {
        for (int k : subs[c]) {
            if (sub_id[k] < 0) {
                sub_id[k] = (int)op.sub_start.size();
                const ClusterNode& C = P.clusters[k];
                op.sub_start.push_back(C.start);
                op.sub_size.push_back(C.size);
                for (int v = C.start; v < C.start + C.size; ++v)
                    for (int e = op.h_vt_ptr[v]; e < op.h_vt_ptr[v + 1]; ++e) {
                        const int t = op.h_vt_idx[e] >> 2;
                        if (stamp[t] != sub_id[k]) {
                            stamp[t] = sub_id[k];
                            tets.push_back(t);
                        }
                    }
                op.sub_tet_ptr.push_back((int)tets.size());
            }
            op.sub_of_cluster.push_back(sub_id[k]);
        }
        op.sub_of_cluster_ptr[c + 1] = (int)op.sub_of_cluster.size();
    }
    return RT_EVALUATOR(op, tables(op, tets, err));
}

static int launch_rows(Operator& op, const std::vector<RowItem>& items, float* out, cudaStream_t s, std::string& err)
{
    if (items.empty()) return RT_OK;
    RowItem* d = nullptr;
    RT_CUDA_TRY(cudaMallocAsync((void**)&d, sizeof(RowItem) * items.size(), s));
    RT_CUDA_TRY(cudaMemcpyAsync(d, items.data(), sizeof(RowItem) * items.size(), cudaMemcpyHostToDevice, s));
    int sums = 0;
    for (const RowItem& it : items) sums = std::max(sums, it.nrow * op.sub_size[it.sub]);
    for (size_t k0 = 0; k0 < items.size(); k0 += (size_t)1 << 30) {
        const int n = (int)std::min<size_t>(items.size() - k0, (size_t)1 << 30);
        const int rc = RT_EVALUATOR(op, rows(op, d + k0, n, sums, out, s, err));
        if (rc) return rc;
    }
    RT_CUDA_TRY(cudaFreeAsync(d, s));
    return RT_OK;
}

// ---------------------------------------------------------------------------
// ACA of the admissible blocks (rt_aca.cuh) and the packing of its terms
// ---------------------------------------------------------------------------
namespace {

// repack converged blocks into V^T [G][r][n] and U^T [G][r][m] in the final storage type
template <class T>
__device__ __forceinline__ T to_store(float x);
template <>
__device__ __forceinline__ float to_store<float>(float x) { return x; }
template <>
__device__ __forceinline__ __nv_bfloat16 to_store<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }
template <>
__device__ __forceinline__ __half to_store<__half>(float x) { return __float2half_rn(x); }

struct PackItem {
    int b;          // far block id (ACA numbering)
    int r, m, n;
    int64_t voff_dst, uoff_dst;   // element offsets of the block's V^T and U^T in the final storage
    int c0, c1;     // chunk range [c0, c1) in the chunk array
};

// Each rank-1 term u v^T is stored as (s u)(v / s) with s chosen so that both
// factors have the same largest magnitude (s = 1 for FP32): the product is
// unchanged and 16-bit storage keeps both factors away from the subnormals.
// With `lo` set, each scaled value x is stored as the 16-bit high part
// h = round(x) in dst and the 16-bit remainder round(x - h) in lo.
template <class T>
__device__ __forceinline__ void store_split(T* dst, T* lo, int64_t i, float x)
{
    const T h = to_store<T>(x);
    dst[i] = h;
    if (lo) lo[i] = to_store<T>(x - (float)h);
}
// blockIdx.y splits a block's terms.  FP32 terms are copied as they are, flat
// over (term, group, column) with 16-byte accesses on the V side; for 16-bit storage
// a warp takes one (term, group) and scales it.  Bound by memory: the terms are
// read once and written once (32^3 x 16 groups, 19 GB: 11.5 ms with a CTA per term
// and its threads on one group's 64 values at a time, 9.5 ms this way).
template <class T>
__global__ void __launch_bounds__(256) aca_pack(AcaDev D, const PackItem* items, int nitems, const Chunk* chunks, T* dst, T* lo)
{
    const int lane = threadIdx.x & 31, warp = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int warps = gridDim.y * (blockDim.x >> 5);
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const PackItem p = items[it];
        const int m4 = round4(p.m), n4 = round4(p.n), n8 = round8(p.n);
        if constexpr (sizeof(T) == 4) {
            const int64_t* toff = D.toff + (int64_t)p.b * D.rmax;
            const int tid = blockIdx.y * blockDim.x + threadIdx.x, nth = gridDim.y * blockDim.x;
            // 32-bit counters over at most 2^30 elements at a time
            const int nq = n4 >> 2, per = D.G * nq;   // float4s of one term's V
            for (int l0 = 0, lc; l0 < p.r; l0 += lc) {
                lc = min(p.r - l0, max(1, (1 << 30) / per));
#pragma unroll 4
                for (int e = tid; e < lc * per; e += nth) {
                    const int lr = e / per, k = e - lr * per, g = k / nq, l = l0 + lr;
                    const float4 x = reinterpret_cast<const float4*>(D.pool + toff[l] + (int64_t)D.G * m4)[k];
                    *reinterpret_cast<float4*>(dst + p.voff_dst + ((int64_t)g * p.r + l) * n8 + 4 * (k - g * nq)) = x;
                }
            }
            for (int c = p.c0; c < p.c1; ++c) {
                const Chunk ch = chunks[c];
                const int pu = D.G * ch.m;
#pragma unroll 4
                for (int e = tid; e < p.r * pu; e += nth) {
                    const int l = e / pu, k = e - l * pu, g = k / ch.m, i = k - g * ch.m;
                    dst[p.uoff_dst + ch.off + ((int64_t)g * p.r + l) * ch.m8 + i] = D.pool[toff[l] + (int64_t)g * m4 + ch.rbeg + i];
                }
            }
            continue;
        }
        for (int k = warp; k < p.r * D.G; k += warps) {
            const int l = k / D.G, g = k - l * D.G;
            const float* u = D.pool + D.toff[(int64_t)p.b * D.rmax + l] + (int64_t)g * m4;
            const float* v = D.pool + D.toff[(int64_t)p.b * D.rmax + l] + (int64_t)D.G * m4 + (int64_t)g * n4;
            float su = 1.f;
            if (sizeof(T) == 2) {
                float mu = 0.f, mv = 0.f;
                for (int i = lane; i < p.m; i += 32) mu = fmaxf(mu, fabsf(u[i]));
                for (int j = lane; j < p.n; j += 32) mv = fmaxf(mv, fabsf(v[j]));
                for (int o = 16; o > 0; o >>= 1) {
                    mu = fmaxf(mu, __shfl_xor_sync(0xffffffffu, mu, o));
                    mv = fmaxf(mv, __shfl_xor_sync(0xffffffffu, mv, o));
                }
                if (mu > 0.f && mv > 0.f) su = sqrtf(mv / mu);
            }
            const float sv = 1.f / su;
            const int64_t vd = p.voff_dst + ((int64_t)g * p.r + l) * n8;
            for (int j = lane; j < p.n; j += 32) store_split<T>(dst, lo, vd + j, sv * v[j]);
            for (int c = p.c0; c < p.c1; ++c) {
                const Chunk ch = chunks[c];
                const int64_t ud = p.uoff_dst + ch.off + ((int64_t)g * p.r + l) * ch.m8;
                for (int i = lane; i < ch.m; i += 32) store_split<T>(dst, lo, ud + i, su * u[ch.rbeg + i]);
            }
        }
    }
}

}  // namespace

int assemble_hmatrix(Operator& op, cudaStream_t s, std::string& err)
{
    int rc;
    const int G = op.G;
    const std::vector<FarBlock>& farb = op.plan.far_blocks;
    const int nfar = (int)farb.size();
    const int rmax = op.rank_max;
    cudaEvent_t ev0, ev1;
    cudaEventCreate(&ev0);
    cudaEventCreate(&ev1);
    cudaEventRecord(ev0, s);

    std::vector<int> final_status(nfar, ACA_DENSE), final_rank(nfar, 0);
    int64_t aca_steps = 0;
    AcaDev D{};
    std::vector<void*> tmp;   // freed at the end
    int64_t scratch = 0;      // bytes of ACA scratch held now (tmp, pool, dot lists)
    auto note_peak = [&](int64_t extra) {
        op.info.peak_bytes = std::max<int64_t>(op.info.peak_bytes, op.info.device_bytes + op.eval_bytes + scratch + extra);
    };
    auto talloc = [&](void** p, size_t bytes) -> int {
        cudaError_t e = cudaMallocAsync(p, bytes ? bytes : 1, s);
        if (e != cudaSuccess) {
            err = std::string("cudaMalloc (ACA scratch): ") + cudaGetErrorString(e);
            return RT_ENOMEM;
        }
        tmp.push_back(*p);
        scratch += (int64_t)(bytes ? bytes : 1);
        note_peak(0);
        return RT_OK;
    };
    auto cleanup = [&]() {
        for (void* p : tmp) cudaFreeAsync(p, s);
        tmp.clear();
    };
    float* pool = nullptr;
    int64_t pool_cap = 0;
    float ms = 0.f, ms_pack = 0.f;
    const int esz = op.far_prec == RT_PREC_F32 ? 4 : 2;
    const bool split = op.refine && op.far_prec != RT_PREC_F32;

    // ---- waves: consecutive runs of far blocks whose ACA terms (estimated at
    // kPoolTerms terms per block) take at most kWaveBytes of FP32 scratch.  Each
    // wave is approximated, packed into the far storage and its scratch freed
    // before the next starts, which bounds the assembly's memory peak.
    const int64_t kWaveBytes = op.wave_bytes;
    std::vector<int> wave_start(1, 0);
    {
        double acc = 0.0;
        for (int b = 0; b < nfar; ++b) {
            const double est = 4.0 * G * (double)(farb[b].m + farb[b].n) * (double)kPoolTerms;
            if (acc > 0.0 && acc + est > (double)kWaveBytes) {
                wave_start.push_back(b);
                acc = 0.0;
            }
            acc += est;
        }
        wave_start.push_back(nfar);
    }
    const int nwaves = (int)wave_start.size() - 1;
    op.info.aca_waves = nfar > 0 ? nwaves : 0;
    int nw_max = 0;
    int64_t summ_max = 0;
    for (int w = 0; w < nwaves; ++w) {
        int64_t sm = 0;
        for (int b = wave_start[w]; b < wave_start[w + 1]; ++b) {
            sm += farb[b].m;
        }
        nw_max = std::max(nw_max, wave_start[w + 1] - wave_start[w]);
        summ_max = std::max(summ_max, sm);
    }

    // final far storage layout, filled wave by wave
    op.far_blocks.clear();
    op.dense_blocks = op.plan.near_blocks;
    op.rank.clear();
    op.far_v_off.clear();
    op.far_u_off.clear();
    op.far_chunks.clear();
    op.far_chunk_ptr.assign(1, 0);
    std::vector<int> far_src;   // ACA block id of each stored far block
    int64_t far_elems = 0;
    if (nwaves > 1) {
        // address range for the largest possible far field: every block at the
        // rank where dense storage becomes cheaper
        int64_t bound = 0;
        std::vector<Chunk> tmpc;
        for (int b = 0; b < nfar; ++b) {
            const FarBlock& fb = farb[b];
            const int64_t rcap = std::min<int64_t>(rmax, (int64_t)fb.m * fb.n / (fb.m + fb.n) + 1);
            tmpc.clear();
            bound += (int64_t)G * rcap * ((int64_t)round8(fb.n) + block_chunks(op.plan, fb.row0, fb.m, 1, tmpc));
        }
        if ((rc = growbuf_reserve(op.far_buf, (size_t)bound * esz, op.device, err))) return rc;
        if (split && (rc = growbuf_reserve(op.far_lo_buf, (size_t)bound * esz, op.device, err))) return rc;
    }
    if (nfar > 0) {
        D.G = G;
        D.rmax = rmax;
        D.eps = op.aca_eps;
#define TA(ptr, bytes)                                       \
    do {                                                     \
        if ((rc = talloc((void**)&(ptr), (bytes)))) {        \
            cleanup();                                       \
            return rc;                                       \
        }                                                    \
    } while (0)
        // per-block state, sized for the largest wave and indexed by the
        // block's position in its wave
        FarBlock* d_blk;
        TA(d_blk, sizeof(FarBlock) * nw_max);
        TA(D.istar, sizeof(int) * nw_max);
        TA(D.rank, sizeof(int) * nw_max);
        TA(D.steps, sizeof(int) * nw_max);
        TA(D.status, sizeof(int) * nw_max);
        TA(D.norm2, sizeof(double) * nw_max * G);
        TA(D.wscale, sizeof(float) * nw_max * G);
        TA(D.toff, sizeof(int64_t) * nw_max * rmax);
        TA(D.used, summ_max);
        TA(D.used_off, sizeof(int64_t) * nw_max);
        int *d_order, *d_sub_ptr, *d_sub_of, *d_ctl;
        TA(d_order, sizeof(int) * nw_max);
        TA(d_sub_ptr, sizeof(int) * op.sub_of_cluster_ptr.size());
        TA(d_sub_of, sizeof(int) * op.sub_of_cluster.size());
        TA(d_ctl, 4 * sizeof(int));   // terms taken from the pool (8 bytes), next block, most steps
        D.blk = d_blk;
        D.order = d_order;
        D.sub_ptr = d_sub_ptr;
        D.sub_of = d_sub_of;
        D.pool_used = (unsigned long long*)d_ctl;
        D.next = d_ctl + 2;
        D.max_steps = d_ctl + 3;
        RT_CUDA_TRY(cudaMemcpyAsync(d_sub_ptr, op.sub_of_cluster_ptr.data(), sizeof(int) * op.sub_of_cluster_ptr.size(),
                                    cudaMemcpyHostToDevice, s));
        RT_CUDA_TRY(cudaMemcpyAsync(d_sub_of, op.sub_of_cluster.data(), sizeof(int) * op.sub_of_cluster.size(),
                                    cudaMemcpyHostToDevice, s));
        int widest = 1;
        for (int c : op.sub_size) widest = std::max(widest, c);
        std::vector<int> h_status_buf((size_t)nw_max * 2);
        int* h_status = h_status_buf.data();
        const std::vector<float> ones((size_t)nw_max * G, 1.0f);
        cudaEvent_t pk0, pk1;
        cudaEventCreate(&pk0);
        cudaEventCreate(&pk1);

        for (int w = 0; w < nwaves; ++w) {
            const int w0 = wave_start[w], nb = wave_start[w + 1] - w0;
            const FarBlock* fw = farb.data() + w0;
            std::vector<int64_t> used_off(nb);
            int64_t sum_m = 0;
            for (int b = 0; b < nb; ++b) {
                used_off[b] = sum_m;
                sum_m += fw[b].m;
            }
            RT_CUDA_TRY(cudaMemcpyAsync(d_blk, fw, sizeof(FarBlock) * nb, cudaMemcpyHostToDevice, s));
            RT_CUDA_TRY(cudaMemsetAsync(D.istar, 0, sizeof(int) * nb, s));
            RT_CUDA_TRY(cudaMemsetAsync(D.rank, 0, sizeof(int) * nb, s));
            RT_CUDA_TRY(cudaMemsetAsync(D.steps, 0, sizeof(int) * nb, s));
            RT_CUDA_TRY(cudaMemsetAsync(D.status, 0, sizeof(int) * nb, s));
            RT_CUDA_TRY(cudaMemsetAsync(D.norm2, 0, sizeof(double) * nb * G, s));
            RT_CUDA_TRY(cudaMemcpyAsync(D.wscale, ones.data(), sizeof(float) * nb * G, cudaMemcpyHostToDevice, s));
            RT_CUDA_TRY(cudaMemsetAsync(D.used, 0, sum_m, s));
            RT_CUDA_TRY(cudaMemcpyAsync(D.used_off, used_off.data(), sizeof(int64_t) * nb, cudaMemcpyHostToDevice, s));
            std::vector<int> h_rank(nb, 0), status(nb, ACA_ACTIVE);

            // term pool of this wave, grown if needed
            int64_t one_term = 0;
            for (int b = 0; b < nb; ++b) one_term += aca_term_size(G, fw[b].m, fw[b].n);
            pool_cap = pool_first(one_term);
            if (cudaMallocAsync((void**)&pool, sizeof(float) * pool_cap, s) != cudaSuccess) {
                cleanup();
                err = "cudaMalloc (ACA pool) failed";
                return RT_ENOMEM;
            }
            D.pool = pool;
            scratch += (int64_t)sizeof(float) * pool_cap;
            note_peak(0);

            // largest blocks first, so that none starts late (counting sort by m + n)
            {
                int most = 0;
                for (int b = 0; b < nb; ++b) most = std::max(most, fw[b].m + fw[b].n);
                std::vector<int> first(most + 2, 0), order(nb);
                for (int b = 0; b < nb; ++b) first[most - (fw[b].m + fw[b].n) + 1]++;
                for (int k = 0; k <= most; ++k) first[k + 1] += first[k];
                for (int b = 0; b < nb; ++b) order[first[most - (fw[b].m + fw[b].n)]++] = b;
                RT_CUDA_TRY(cudaMemcpyAsync(d_order, order.data(), sizeof(int) * nb, cudaMemcpyHostToDevice, s));
            }
            RT_CUDA_TRY(cudaMemsetAsync(d_ctl, 0, 4 * sizeof(int), s));
            D.nb = nb;
            for (bool more = true; more;) {
                D.pool_cap = pool_cap;
                RT_CUDA_TRY(cudaMemsetAsync(D.next, 0, sizeof(int), s));
                if ((rc = RT_EVALUATOR(op, aca(op, D, widest, s, err)))) {
                    cudaFreeAsync(pool, s);
                    cleanup();
                    return rc;
                }
                int ctl[4];
                RT_CUDA_TRY(cudaMemcpyAsync(h_status, D.status, sizeof(int) * nb, cudaMemcpyDeviceToHost, s));
                RT_CUDA_TRY(cudaMemcpyAsync(h_status + nb, D.rank, sizeof(int) * nb, cudaMemcpyDeviceToHost, s));
                RT_CUDA_TRY(cudaMemcpyAsync(ctl, d_ctl, sizeof(ctl), cudaMemcpyDeviceToHost, s));
                RT_CUDA_TRY(cudaStreamSynchronize(s));
                more = false;
                int64_t need = 0;   // one more term for every block that is still active
                for (int b = 0; b < nb; ++b) {
                    status[b] = h_status[b];
                    h_rank[b] = h_status[nb + b];
                    if (status[b] == ACA_ACTIVE) {
                        more = true;
                        need += aca_term_size(G, fw[b].m, fw[b].n);
                    }
                }
                if (!more) {
                    aca_steps += ctl[3];
                    break;
                }
                // the pool ran out: a larger one, and the active blocks go on
                const int64_t ncap = pool_grown(pool_cap, need);
                float* np = nullptr;
                if (cudaMallocAsync((void**)&np, sizeof(float) * ncap, s) != cudaSuccess) {
                    cudaFreeAsync(pool, s);
                    cleanup();
                    err = "cudaMalloc (ACA pool growth) failed";
                    return RT_ENOMEM;
                }
                RT_CUDA_TRY(cudaMemcpyAsync(np, pool, sizeof(float) * pool_cap, cudaMemcpyDeviceToDevice, s));
                note_peak((int64_t)sizeof(float) * ncap);   // old and new pool both live here
                scratch += (int64_t)sizeof(float) * (ncap - pool_cap);
                cudaFreeAsync(pool, s);
                const unsigned long long taken = (unsigned long long)pool_cap;
                RT_CUDA_TRY(cudaMemcpyAsync(D.pool_used, &taken, sizeof(taken), cudaMemcpyHostToDevice, s));
                pool = np;
                pool_cap = ncap;
                D.pool = pool;
            }
            // ---- this wave's blocks: stored low rank, all-zero, or dense ------
            const int64_t elems0 = far_elems;
            const int k0 = (int)op.far_blocks.size();
            for (int b = 0; b < nb; ++b) {
                final_status[w0 + b] = status[b] == ACA_ACTIVE ? ACA_DENSE : status[b];
                final_rank[w0 + b] = h_rank[b];
                if (final_status[w0 + b] == ACA_DONE && h_rank[b] > 0) {
                    const FarBlock& fb = fw[b];
                    const int r = h_rank[b];
                    op.far_blocks.push_back(fb);
                    op.rank.push_back(r);
                    far_src.push_back(b);
                    op.far_v_off.push_back(far_elems);
                    far_elems += (int64_t)G * r * round8(fb.n);
                    op.far_u_off.push_back(far_elems);
                    far_elems += block_chunks(op.plan, fb.row0, fb.m, (int64_t)G * r, op.far_chunks);
                    op.far_chunk_ptr.push_back((int)op.far_chunks.size());
                } else if (final_status[w0 + b] == ACA_DONE) {
                    // an all-zero block: nothing to store
                } else {
                    op.dense_blocks.push_back(fw[b]);
                    op.n_fallback++;
                }
            }
            const int k1 = (int)op.far_blocks.size();
            // ---- storage for the new far blocks, then pack them -----------------
            if (nwaves == 1 && k1 > 0) {
                char *d = nullptr, *dl = nullptr;
                if ((rc = dev_alloc(op, &d, (size_t)far_elems * esz, err)) ||
                    (split && (rc = dev_alloc(op, &dl, (size_t)far_elems * esz, err)))) {
                    cudaFreeAsync(pool, s);
                    cleanup();
                    return rc;
                }
                op.d_far = d;
                op.d_far_lo = dl;
            } else if (nwaves > 1 && far_elems > elems0) {
                const size_t before = op.far_buf.mapped;
                if ((rc = growbuf_grow(op.far_buf, (size_t)far_elems * esz, err)) ||
                    (split && (rc = growbuf_grow(op.far_lo_buf, (size_t)far_elems * esz, err)))) {
                    cudaFreeAsync(pool, s);
                    cleanup();
                    return rc;
                }
                op.info.device_bytes += (int64_t)(op.far_buf.mapped - before) * (split ? 2 : 1);
                op.d_far = (void*)op.far_buf.base;
                op.d_far_lo = split ? (void*)op.far_lo_buf.base : nullptr;
            }
            if (k1 > k0) {
                char* base = (char*)op.d_far;
                char* base_lo = (char*)op.d_far_lo;
                RT_CUDA_TRY(cudaMemsetAsync(base + elems0 * esz, 0, (size_t)(far_elems - elems0) * esz, s));
                if (base_lo) RT_CUDA_TRY(cudaMemsetAsync(base_lo + elems0 * esz, 0, (size_t)(far_elems - elems0) * esz, s));
                note_peak(0);   // packed far field next to this wave's pool
                std::vector<PackItem> items;
                for (int k = k0; k < k1; ++k)
                    items.push_back({far_src[k], op.rank[k], op.far_blocks[k].m, op.far_blocks[k].n, op.far_v_off[k],
                                     op.far_u_off[k], op.far_chunk_ptr[k], op.far_chunk_ptr[k + 1]});
                PackItem* d_items = nullptr;
                Chunk* d_chunks = nullptr;
                const int c0 = op.far_chunk_ptr[k0], nc = op.far_chunk_ptr[k1] - c0;
                RT_CUDA_TRY(cudaMallocAsync((void**)&d_items, sizeof(PackItem) * items.size(), s));
                RT_CUDA_TRY(cudaMallocAsync((void**)&d_chunks, sizeof(Chunk) * op.far_chunks.size(), s));
                RT_CUDA_TRY(cudaMemcpyAsync(d_items, items.data(), sizeof(PackItem) * items.size(),
                                            cudaMemcpyHostToDevice, s));
                RT_CUDA_TRY(cudaMemcpyAsync(d_chunks + c0, op.far_chunks.data() + c0, sizeof(Chunk) * nc,
                                            cudaMemcpyHostToDevice, s));
                const dim3 grid((unsigned)std::min<size_t>(items.size(), 152 * 64), items.size() < 152 * 8 ? 8 : 1);
                const int ni = (int)items.size();
                cudaEventRecord(pk0, s);
                if (op.far_prec == RT_PREC_F32)
                    aca_pack<float><<<grid, 256, 0, s>>>(D, d_items, ni, d_chunks, (float*)base, nullptr);
                else if (op.far_prec == RT_PREC_BF16)
                    aca_pack<__nv_bfloat16><<<grid, 256, 0, s>>>(D, d_items, ni, d_chunks, (__nv_bfloat16*)base,
                                                                 (__nv_bfloat16*)base_lo);
                else aca_pack<__half><<<grid, 256, 0, s>>>(D, d_items, ni, d_chunks, (__half*)base, (__half*)base_lo);
                cudaEventRecord(pk1, s);
                RT_CUDA_TRY(cudaGetLastError());
                cudaFreeAsync(d_items, s);
                cudaFreeAsync(d_chunks, s);
                RT_CUDA_TRY(cudaEventSynchronize(pk1));
                float t = 0.f;
                cudaEventElapsedTime(&t, pk0, pk1);
                ms_pack += t;
            }
            cudaFreeAsync(pool, s);
            scratch -= (int64_t)sizeof(float) * pool_cap;
            pool = nullptr;
        }
        cudaEventDestroy(pk0);
        cudaEventDestroy(pk1);
#undef TA
    }
    cleanup();
    scratch = 0;
    op.n_far = (int)op.far_blocks.size();
    op.n_near = (int)op.dense_blocks.size();
    cudaEventRecord(ev1, s);
    cudaEventSynchronize(ev1);
    cudaEventElapsedTime(&ms, ev0, ev1);
    op.info.ms_aca = ms - ms_pack;
    op.info.ms_pack = ms_pack;
    op.info.aca_steps = aca_steps;

    // ---- dense blocks (near leaves and fallbacks): per leaf chunk A^T [G][n][m8]
    cudaEventRecord(ev0, s);
    int64_t near_elems = 0;
    op.dense_off.assign(op.n_near, 0);
    op.dense_chunks.clear();
    op.dense_chunk_ptr.assign(1, 0);
    for (int k = 0; k < op.n_near; ++k) {
        const FarBlock& fb = op.dense_blocks[k];
        op.dense_off[k] = near_elems;
        near_elems += block_chunks(op.plan, fb.row0, fb.m, (int64_t)G * fb.n, op.dense_chunks);
        op.dense_chunk_ptr.push_back((int)op.dense_chunks.size());
    }
    if (op.n_near > 0) {
        if ((rc = dev_alloc(op, &op.d_near, (size_t)near_elems, err))) return rc;
        RT_CUDA_TRY(cudaMemsetAsync(op.d_near, 0, sizeof(float) * (size_t)near_elems, s));
        std::vector<RowItem> ritems;
        for (int k = 0; k < op.n_near; ++k) {
            const FarBlock& fb = op.dense_blocks[k];
            for (int c = op.dense_chunk_ptr[k]; c < op.dense_chunk_ptr[k + 1]; ++c) {
                const Chunk& ch = op.dense_chunks[c];
                for (int e = op.sub_of_cluster_ptr[fb.sc]; e < op.sub_of_cluster_ptr[fb.sc + 1]; ++e) {
                    const int sb = op.sub_of_cluster[e];
                    const int rows = rows_per_item(group_chunk(op), op.sub_size[sb]);
                    for (int ii = 0; ii < ch.m; ii += rows) {
                        RowItem it{};
                        it.i = fb.row0 + ch.rbeg + ii;
                        it.nrow = std::min(rows, ch.m - ii);
                        it.sub = sb;
                        it.out = op.dense_off[k] + ch.off + ii + (int64_t)(op.sub_start[sb] - fb.col0) * ch.m8;
                        it.gs = (int64_t)fb.n * ch.m8;
                        it.js = ch.m8;
                        ritems.push_back(it);
                    }
                }
            }
        }
        note_peak((int64_t)(sizeof(RowItem) * ritems.size()));   // near blocks, tables and items
        if ((rc = launch_rows(op, ritems, op.d_near, s, err))) return rc;
        for (int k = 0; k < op.n_near; ++k)
            op.info.entries_evaluated += (int64_t)op.dense_blocks[k].m * op.dense_blocks[k].n;
    }
    RT_CUDA_TRY(cudaStreamSynchronize(s));
    cudaEventRecord(ev1, s);
    cudaEventSynchronize(ev1);
    cudaEventElapsedTime(&ms, ev0, ev1);
    op.info.ms_near = ms;
    cudaEventDestroy(ev0);
    cudaEventDestroy(ev1);

    // ---- statistics ------------------------------------------------------------
    int64_t stored = 0, rsum = 0, rmin = INT64_MAX, rmx = 0;
    for (int k = 0; k < op.n_near; ++k) stored += (int64_t)op.dense_blocks[k].m * op.dense_blocks[k].n;
    for (int k = 0; k < op.n_far; ++k) {
        stored += (int64_t)op.rank[k] * (op.far_blocks[k].m + op.far_blocks[k].n);
        rsum += op.rank[k];
        rmin = std::min<int64_t>(rmin, op.rank[k]);
        rmx = std::max<int64_t>(rmx, op.rank[k]);
    }
    op.info.stored_entries = stored;
    op.info.rank_sum = rsum;
    op.info.rank_min = op.n_far ? rmin : 0;
    op.info.rank_max = rmx;
    for (int b = 0; b < nfar; ++b) op.info.entries_evaluated += (int64_t)final_rank[b] * (farb[b].m + farb[b].n);
    return RT_OK;
}


// ---------------------------------------------------------------------------
// Rows of the surface-to-volume matrix Sbar^E_{i,l} (Section 2, last
// paragraph): the emitter source with Q0 replaced by the P1 hat function of
// emitter vertex l.  Each quadrature value of a triangle is split over the
// triangle's three vertices by its barycentric weights; a source point that is
// a vertex of the triangle gives that vertex the limit (angle)/(8 pi).  One CTA
// per row, threads over the emitter triangles, the row [G][L] accumulated in
// shared memory (float atomics: the summation order is not fixed).
// col_of[v] = column (surface tree order) of tree vertex v, -1 off the emitter.
// out[g * gstride + (i - row0) * L + l], rows i in [row0, row0 + nrows).
// ---------------------------------------------------------------------------
template <int MG>
__global__ void __launch_bounds__(256) srcop_rows_kernel(KernelParams P, int n_emit, const int4* __restrict__ emit,
                                                         const int* __restrict__ col_of, int L, int row0, int nrows,
                                                         float* __restrict__ out, int64_t gstride)
{
    extern __shared__ float srow[];   // [G][L]
    const int G = P.G;
    const float inv4pi = (float)(1.0 / (4.0 * kPi));
    for (int r = blockIdx.x; r < nrows; r += gridDim.x) {
        const int i = row0 + r;
        __syncthreads();
        for (int k = threadIdx.x; k < G * L; k += blockDim.x) srow[k] = 0.f;
        __syncthreads();
        const Vec3<float> xi = load_xyz<float>(P, i);
        Vec3<float> xb = xi;
        bool on_wall = false;
        if (P.has_wall) {
            xb = mirror_point<float>(P, xi);
            on_wall = dist2<float>(xi, xb) <= 1e-20f;
        }
        for (int e = threadIdx.x; e < n_emit; e += blockDim.x) {
            const int4 tv = emit[e];
            const int cl[3] = {col_of[tv.x], col_of[tv.y], col_of[tv.z]};
            const Vec3<float> V0 = load_xyz<float>(P, tv.x), V1 = load_xyz<float>(P, tv.y),
                              V2 = load_xyz<float>(P, tv.z);
            const Vec3<float> e1 = {V1.x - V0.x, V1.y - V0.y, V1.z - V0.z};
            const Vec3<float> e2 = {V2.x - V0.x, V2.y - V0.y, V2.z - V0.z};
            Vec3<float> nn = {e1.y * e2.z - e1.z * e2.y, e1.z * e2.x - e1.x * e2.z, e1.x * e2.y - e1.y * e2.x};
            const float a2 = sqrtf(nn.x * nn.x + nn.y * nn.y + nn.z * nn.z);
            nn.x /= a2;
            nn.y /= a2;
            nn.z /= a2;
            const float area = 0.5f * a2;
            const Vec3<float> cen = {(V0.x + V1.x + V2.x) / 3.f, (V0.y + V1.y + V2.y) / 3.f, (V0.z + V1.z + V2.z) / 3.f};
            float diam2 = fmaxf(fmaxf(dist2<float>(V0, V1), dist2<float>(V0, V2)), dist2<float>(V1, V2));
            const int vloc = tv.x == i ? 0 : (tv.y == i ? 1 : (tv.z == i ? 2 : -1));
            float a[3][MG];
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int g = 0; g < MG; ++g) a[k][g] = 0.f;
            for (int term = 0; term < 2 + P.n_extra; ++term) {
                if (term == 1 && !P.has_wall) continue;
                Vec3<float> src;
                float scale;
                term_source<float>(P, term, xi, xb, src, scale);
                const bool at_x = term == 0 || (term == 1 ? on_wall : dist2<float>(xi, src) <= 1e-20f);
                if (vloc >= 0 && at_x) {
                    const Vec3<float> A = vloc == 0 ? V0 : (vloc == 1 ? V1 : V2);
                    const Vec3<float> B = vloc == 0 ? V1 : (vloc == 1 ? V2 : V0);
                    const Vec3<float> Cc = vloc == 0 ? V2 : (vloc == 1 ? V0 : V1);
                    const Vec3<float> u = {B.x - A.x, B.y - A.y, B.z - A.z}, v = {Cc.x - A.x, Cc.y - A.y, Cc.z - A.z};
                    float cs = (u.x * v.x + u.y * v.y + u.z * v.z) /
                               sqrtf((u.x * u.x + u.y * u.y + u.z * u.z) * (v.x * v.x + v.y * v.y + v.z * v.z));
                    cs = fminf(1.f, fmaxf(-1.f, cs));
                    const float lim = scale * acosf(cs) * (float)(1.0 / (8.0 * kPi));
#pragma unroll
                    for (int g = 0; g < MG; ++g) a[vloc][g] += lim;
                    continue;
                }
                const float sd = (src.x - V0.x) * nn.x + (src.y - V0.y) * nn.y + (src.z - V0.z) * nn.z;
                if (!(sd < 0.f)) continue;
                const float cm = -sd;
                const bool nearp = dist2<float>(src, cen) < 4.f * diam2;
                const int q0 = nearp ? 3 : 0, nq = nearp ? 7 : 3;
                for (int q = 0; q < nq; ++q) {
                    const float b[3] = {(float)c_tri_b[3 * (q0 + q)], (float)c_tri_b[3 * (q0 + q) + 1],
                                        (float)c_tri_b[3 * (q0 + q) + 2]};
                    const Vec3<float> y = {b[0] * V0.x + b[1] * V1.x + b[2] * V2.x, b[0] * V0.y + b[1] * V1.y + b[2] * V2.y,
                                           b[0] * V0.z + b[1] * V1.z + b[2] * V2.z};
                    const float r2 = dist2<float>(src, y);
                    const float tau = term_depth<float>(P, term, xi, src, y);
                    const float geo = scale * area * (float)c_tri_w[q0 + q] * cm * cm / (r2 * r2) * inv4pi;
#pragma unroll
                    for (int g = 0; g < MG; ++g) {
                        if (g < G) {
                            const float v = geo * expf(-P.cf[g] * tau);
#pragma unroll
                            for (int k = 0; k < 3; ++k) a[k][g] += v * b[k];
                        }
                    }
                }
            }
#pragma unroll
            for (int g = 0; g < MG; ++g)
                if (g < G)
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        if (cl[k] >= 0) atomicAdd(srow + g * L + cl[k], a[k][g]);
        }
        __syncthreads();
        for (int k = threadIdx.x; k < G * L; k += blockDim.x) {
            const int g = k / L, l = k - g * L;
            out[g * gstride + (int64_t)r * L + l] = srow[k];
        }
    }
}

int srcop_eval_rows(Operator& op, const int* col_of, int L, int row0, int nrows, float* out, int64_t gstride,
                    cudaStream_t s, std::string& err)
{
    const size_t smem = sizeof(float) * (size_t)op.G * L;
    if (smem > 200 * 1024) {
        err = "surface-to-volume operator: G x L too large for one row in shared memory";
        return RT_EINVAL;
    }
    const int grid = std::max(1, std::min(nrows, 152 * 8));
#define RT_SRC_ROWS(MG)                                                                                        \
    do {                                                                                                       \
        RT_CUDA_TRY(cudaFuncSetAttribute(srcop_rows_kernel<MG>, cudaFuncAttributeMaxDynamicSharedMemorySize,   \
                                         (int)smem));                                                          \
        srcop_rows_kernel<MG><<<grid, 256, smem, s>>>(op.kp, op.n_emit, op.d_emit, col_of, L, row0, nrows, out, \
                                                      gstride);                                                \
    } while (0)
    if (op.G <= 1) RT_SRC_ROWS(1);
    else if (op.G <= 4) RT_SRC_ROWS(4);
    else if (op.G <= 8) RT_SRC_ROWS(8);
    else if (op.G <= 16) RT_SRC_ROWS(16);
    else {
        err = "surface-to-volume operator: at most 16 kappa groups";
        return RT_EINVAL;
    }
#undef RT_SRC_ROWS
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
}

// diagnostic: the library's FP32 sin(2 pi x) beside CUDA's sinpif(2x)
__global__ void sin2pi_probe(const float* __restrict__ x, float* __restrict__ lib, float* __restrict__ ref, int64_t n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        lib[i] = sin2pi(x[i]);
        ref[i] = sinpif(2.0f * x[i]);
    }
}

int eval_sin2pi(const float* x, float* lib, float* ref, int64_t n, cudaStream_t s, std::string& err)
{
    if (n <= 0) return RT_OK;
    const int grid = (int)std::min<int64_t>((n + 255) / 256, 152 * 16);
    sin2pi_probe<<<grid, 256, 0, s>>>(x, lib, ref, n);
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
}

}  // namespace rt

