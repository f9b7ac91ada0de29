// rt_rows.cuh -- rows of G over a column cluster and pivot columns of a block,
// FP32, every kappa group of a chunk of MG groups at once.
//
// Row segment (row i, sub-cluster of consecutive tree-order columns): every
// tetrahedron touching the sub-cluster is visited once, and each quadrature
// value feeds the hat functions of its vertices.  With the 4-point rule the
// value at point q reaches vertex q with weight a and the others with b, so a
// tetrahedron's four vertex sums are b S + (a - b) e_q with S = sum e_q: one
// addition per point and group instead of four products.  The vertex sums go
// to shared memory (a pass of tetrahedra at a time) and every column gathers
// its own from a list made once per operator: plain stores and loads in place
// of 4 G shared float atomics per tetrahedron, which are compare-and-swap
// loops that neighbouring tetrahedra contend for.
//
// Bound: instruction issue (FP32 and the special-function unit); the tables
// stay in L2.  Measured on GB300, all launches of one operator build that still
// launched ACA step by step, before (positions and four sines per optical
// depth, shared atomics) and after (rt_aca.cuh has the ACA's figures since):
//   32^3, 16 groups: rows and near blocks 433 -> 152 ms, columns 148 -> 71 ms
//   41^3, 1 group:   rows and near blocks 400 -> 185 ms, columns 454 -> 163 ms
//   box with grid, walls and corners, 1 group (EV_GENERAL): 901 -> 450 ms
// Near blocks alone now: 66 ms (32^3), 80 ms (41^3, 98 before the point loops were
// rolled up and six CTAs ran on an SM).
// Error against the FP64 oracle, every block dense, before (positions, one group scale
// in FP32 everywhere) and after: entries (root mean square) 1.37e-7 -> 1.33e-7, matvec
// 9.8e-8 -> 9.3e-8 (10^3, 1 group, wall z = 0); 1.36e-7 -> 1.33e-7, 1.07e-7 -> 1.00e-7
// (wall x = 1); 1.63e-7 -> 1.40e-7, 1.17e-7 -> 1.15e-7 (8^3, 16 groups).
//
// (tetrahedron, term) pairs whose source point is near (14-point rule) are
// listed in shared memory and worked off with all lanes full.
#pragma once

#include "rt_phase.cuh"
#include "rt_rows.h"

namespace rt {

// add this thread's counts to the work counters (one atomic per warp and counter)
__device__ __forceinline__ void count_work(const KernelParams& P, unsigned terms, unsigned depths)
{
    if (!P.work) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        terms += __shfl_xor_sync(0xffffffffu, terms, o);
        depths += __shfl_xor_sync(0xffffffffu, depths, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(P.work, (unsigned long long)terms);
        atomicAdd(P.work + 1, (unsigned long long)depths);
    }
}

// Threads of a row or ACA kernel's CTA are a launch parameter: 128, or more when
// a problem has too few blocks to fill the chip (eval_threads in rt_rows.h).
// max_threads is the most that the registers of an instance allow; 128-thread
// CTAs then run six (1 and 4 groups), five (8) or four (16) to an SM.
constexpr int max_threads(int mg, int ev) { return ev != EV_PHASE ? (mg <= 16 ? 512 : 256) : (mg <= 4 ? 768 : (mg <= 8 ? 640 : 512)); }

// Shapes of one row pass: TPT tetrahedra per thread (one group: four, so that a
// pass is worth its two barriers), PT = TPT x threads per pass; stage row of a
// tetrahedron padded so that its 16-byte stores fall into different banks.
template <int MG, int EV>
struct RowShape {
    static constexpr int TPT = tets_per_thread(MG, EV);
    static constexpr int RS = MG == 1 ? 4 : 4 * MG + 4;
    static constexpr int TERMS = EV == EV_GENERAL ? 2 + kMaxXTerms : 2;   // most list entries per tetrahedron
    static __host__ __device__ constexpr int list(int nt) { return 2 * TERMS * TPT * nt; }   // two passes
    // shared bytes of nt threads besides the sums
    static __host__ __device__ constexpr int fixed(int nt)
    {
        return TPT * nt * RS * 4 + 4 * TPT * nt * 2 + kRunWords * 4 + list(nt) * 4;
    }
};

// Term t's value at y for a near pair or a general problem (original
// coordinates): weight over r^2, tau.  False: the path is blocked.
template <bool XT>
__device__ __forceinline__ bool general_term(const KernelParams& P, int t, const Vec3<float>& xi, const Vec3<float>& src,
                                             float scale, const Vec3<float>& y, float w0, float& w, float& tau)
{
    const float r2 = dist2<float>(src, y);
    w = scale * w0 / r2;
    if constexpr (XT) {
        tau = term_depth<float>(P, t, xi, src, y);
        return tau < INFINITY;
    } else {
        if (t == 0) {
            tau = optical_depth<float>(P, xi, y);
        } else {
            const Vec3<float> xp = wall_point<float>(P, src, y);
            tau = optical_depth<float>(P, xi, xp) + optical_depth<float>(P, xp, y);
        }
        return true;
    }
}
__device__ __forceinline__ bool term_present(const KernelParams& P, int t) { return t != 1 || P.has_wall; }
// number of terms of the kernel, and the source point and weight of term t
template <bool XT>
__device__ __forceinline__ int term_count(const KernelParams& P)
{
    return XT ? 2 + P.n_extra : 2;
}
template <bool XT>
__device__ __forceinline__ void source_of(const KernelParams& P, int t, const Vec3<float>& xi, Vec3<float>& src, float& scale)
{
    src = xi;
    scale = 1.f;
    if (t == 1) {
        src = mirror_point<float>(P, xi);
        scale = P.R0f;
    }
    if constexpr (XT) {
        if (t > 1) extra_term<float>(P, t - 2, xi, src, scale);
    }
}

// Point q of the 14-point rule of a tetrahedron: coordinates, weight with
// kappa(y), barycentric weights b
template <bool XT>
__device__ __forceinline__ float near_point(const KernelParams& P, const Vec3<float> (&v)[4], float vol, int q, Vec3<float>& y,
                                            float (&b)[4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) b[k] = tet_b<float>(4 + q, k);
    y = {b[0] * v[0].x + b[1] * v[1].x + b[2] * v[2].x + b[3] * v[3].x,
         b[0] * v[0].y + b[1] * v[1].y + b[2] * v[2].y + b[3] * v[3].y,
         b[0] * v[0].z + b[1] * v[1].z + b[2] * v[2].z + b[3] * v[3].z};
    return vol * tet_w<float>(4 + q) * kappa_at<float, XT>(P, y.x, y.y, y.z) * (float)(1.0 / (4.0 * kPi));
}

// ---- row segments ---------------------------------------------------------------
template <int MG, int EV>
struct RowShared {
    using S = RowShape<MG, EV>;
    float* acc;            // [rows][n][MG]
    float* stage;          // [PT][RS]
    uint16_t* ref;         // [4 PT] offsets into stage, sorted by column
    unsigned* run;         // run count, (column << 16 | first ref) ..., end mark
    unsigned* list;        // near pairs: row << 28 | term << 24 | local tetrahedron
    int* cnt;              // length of list
    __device__ RowShared(char* base, int* counter)
    {
        const int nt = blockDim.x;
        stage = (float*)base;
        ref = (uint16_t*)(stage + S::TPT * nt * S::RS);
        run = (unsigned*)(ref + 4 * S::TPT * nt);
        list = run + kRunWords;
        acc = (float*)(list + S::list(nt));
        cnt = counter;
    }
};

// acc[row][column][g] += the listed near pairs (14-point rule), then the list is empty
template <int MG, int EV>
__device__ __noinline__ void near_flush(const KernelParams& P, const SubInfo& sub, const int* __restrict__ sub_tets, int i0,
                                        int g0, RowShared<MG, EV> sh)
{
    using S = RowShape<MG, EV>;
    const int cnt = *sh.cnt;
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
        const unsigned ent = sh.list[e];
        const int r = ent >> 28, t = (ent >> 24) & 15, tet = sub_tets[sub.tet0 + (ent & 0xffffff)];
        const Vec3<float> xi = load_xyz<float>(P, i0 + r);
        Vec3<float> src;
        float scale;
        source_of<EV == EV_GENERAL>(P, t, xi, src, scale);
        const int4 tv = P.tet[tet];
        const int id[4] = {tv.x, tv.y, tv.z, tv.w};
        Vec3<float> v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = load_xyz<float>(P, id[k]);
        const float vol = P.tvol32[tet];
        float* row = sh.stage + threadIdx.x * S::RS;   // this thread's own
        GroupSum<MG> s;
        s.zero();
#pragma unroll
        for (int k = 0; k < 4; ++k) s.store(row + k * MG);
        for (int q = 0; q < 14; ++q) {
            Vec3<float> y;
            float b[4], w, tau;
            const float w0 = near_point<EV == EV_GENERAL>(P, v, vol, q, y, b);
            if (!general_term<EV == EV_GENERAL>(P, t, xi, src, scale, y, w0, w, tau)) continue;
            s.zero();
            s.add(P, g0, w, tau);
#pragma unroll
            for (int k = 0; k < 4; ++k) s.add_to(row + k * MG, b[k]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int col = id[k] - sub.start;
            if ((unsigned)col >= (unsigned)sub.size) continue;
            float* a = sh.acc + ((int64_t)r * sub.size + col) * MG;
            for (int g = 0; g < MG; ++g) atomicAdd(a + g, row[k * MG + g]);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) *sh.cnt = 0;
    __syncthreads();
}

// acc[r][column][g] = sum over the sub-cluster's tetrahedra of the values of rows
// i0 .. i0 + nrow - 1, without the factor c_g.  Called by the whole CTA.
template <int MG, int EV>
__device__ __forceinline__ void row_segment(const KernelParams& P, const SubInfo& sub, const int* __restrict__ sub_tets,
                                            const uint16_t* __restrict__ pass_ref, const unsigned* __restrict__ pass_run,
                                            int i0, int nrow, int g0, const RowShared<MG, EV>& sh, unsigned& n_terms,
                                            unsigned& n_depths)
{
    using S = RowShape<MG, EV>;
    constexpr int RW = (kRunWords + 127) / 128;
    const int tid = threadIdx.x, nth = blockDim.x, PT = S::TPT * nth, list_cap = S::list(nth);
    for (int k = tid; k < nrow * sub.size * MG; k += nth) sh.acc[k] = 0.f;
    if (tid == 0) *sh.cnt = 0;
    __syncthreads();
    const int npass = (sub.ntet + PT - 1) / PT;
    for (int p = 0; p < npass; ++p) {
        // this pass's gather lists: fetched now, stored before the first barrier
        uint2 refs[S::TPT];
        unsigned run_w[RW];
        {
            const uint2* gr = reinterpret_cast<const uint2*>(pass_ref + (int64_t)(sub.pass0 + p) * 4 * PT);
            const unsigned* gw = pass_run + (int64_t)(sub.pass0 + p) * kRunWords;
#pragma unroll
            for (int k = 0; k < S::TPT; ++k) refs[k] = gr[k * nth + tid];
#pragma unroll
            for (int k = 0; k < RW; ++k)
                run_w[k] = k * nth + tid < kRunWords ? gw[k * nth + tid] : 0u;
        }
        for (int r = 0; r < nrow; ++r) {
            const int i = i0 + r;
            const Vec3<float> xi = load_xyz<float>(P, i);
#pragma unroll 1
            for (int tt = 0; tt < S::TPT; ++tt) {
                const int tl = p * PT + tt * nth + tid;
                if (tl >= sub.ntet) break;
                const int tet = sub_tets[sub.tet0 + tl];
                const float4 cen4 = P.tcen[tet];
                const Vec3<float> cen = {cen4.x, cen4.y, cen4.z};
                float* row = sh.stage + (tt * nth + tid) * S::RS;
                GroupSum<MG> sum;
                sum.zero();
                if constexpr (EV == EV_PHASE) {
                    const PhasePoint x = phase_point(P, i);
                    const bool fd = !(dist2<float>(xi, cen) < cen4.w);
                    const bool fr = P.has_wall && !(dist2<float>(mirror_point<float>(P, xi), cen) < cen4.w);
                    if (!fd) sh.list[atomicAdd(sh.cnt, 1)] = ((unsigned)r << 28) | (unsigned)tl;
                    if (P.has_wall && !fr) sh.list[atomicAdd(sh.cnt, 1)] = ((unsigned)r << 28) | (1u << 24) | (unsigned)tl;
                    n_terms += (fd ? 4 : 14) + (P.has_wall ? (fr ? 4 : 14) : 0);
                    n_depths += (fd ? 4 : 14) + (P.has_wall ? 2 * (fr ? 4 : 14) : 0);
#pragma unroll 1
                    for (int q = 0; q < 4; ++q) {
                        const float4 y4 = P.tpt[(int64_t)q * P.T + tet];
                        float4 yc = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (P.sinprod) yc = P.tcos[(int64_t)q * P.T + tet];
                        GroupSum<MG> e;
                        e.zero();
                        float w, tau;
                        if (fd) {
                            phase_direct(P, x, y4, yc, w, tau);
                            e.add(P, g0, w, tau);
                        }
                        if (fr) {
                            phase_reflected(P, x, y4, yc, w, tau);
                            e.add(P, g0, w, tau);
                        }
                        sum.add(e);
                        e.store(row + q * MG);
                    }
                } else {
                    unsigned far = 0u;
                    const int nt = term_count<EV == EV_GENERAL>(P);
                    for (int t = 0; t < nt; ++t) {
                        if (!term_present(P, t)) continue;
                        Vec3<float> src;
                        float scale;
                        source_of<EV == EV_GENERAL>(P, t, xi, src, scale);
                        const int legs = t == 0 ? 1 : (t == 1 ? 2 : P.xkind[t - 2] + 1);
                        const bool nr = dist2<float>(src, cen) < cen4.w;
                        if (nr) sh.list[atomicAdd(sh.cnt, 1)] = ((unsigned)r << 28) | ((unsigned)t << 24) | (unsigned)tl;
                        else far |= 1u << t;
                        n_terms += nr ? 14 : 4;
                        n_depths += (nr ? 14 : 4) * legs;
                    }
#pragma unroll 1
                    for (int q = 0; q < 4; ++q) {
                        const float4 y4 = P.tpt[(int64_t)q * P.T + tet];
                        const Vec3<float> y = {y4.x, y4.y, y4.z};
                        GroupSum<MG> e;
                        e.zero();
#pragma unroll 1
                        for (int t = 0; t < nt; ++t) {
                            if (!(far >> t & 1u)) continue;
                            Vec3<float> src;
                            float scale, w, tau;
                            source_of<EV == EV_GENERAL>(P, t, xi, src, scale);
                            if (general_term<EV == EV_GENERAL>(P, t, xi, src, scale, y, y4.w, w, tau)) e.add(P, g0, w, tau);
                        }
                        sum.add(e);
                        e.store(row + q * MG);
                    }
                }
                if constexpr (MG == 1) {
                    const float bs = kTetB * sum.e;
                    float4 e = *reinterpret_cast<float4*>(row);
                    e = make_float4(fmaf(kTetG, e.x, bs), fmaf(kTetG, e.y, bs), fmaf(kTetG, e.z, bs), fmaf(kTetG, e.w, bs));
                    *reinterpret_cast<float4*>(row) = e;
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) sum.blend(row + q * MG, kTetB, kTetG);
                }
            }
            if (r == 0) {
#pragma unroll
                for (int k = 0; k < S::TPT; ++k) reinterpret_cast<uint2*>(sh.ref)[k * nth + tid] = refs[k];
#pragma unroll
                for (int k = 0; k < RW; ++k)
                    if (k * nth + tid < kRunWords) sh.run[k * nth + tid] = run_w[k];
            }
            __syncthreads();
            // MG lanes per column run
            const int nrun = (int)sh.run[0], g = tid % MG;
            for (int k = tid / MG; k < nrun; k += nth / MG) {
                const unsigned w0 = sh.run[1 + k];
                const int a = w0 & 0xffff, b = sh.run[2 + k] & 0xffff;
                float v = 0.f;
#pragma unroll 4
                for (int e = a; e < b; ++e) v += sh.stage[sh.ref[e] + g];
                sh.acc[((int64_t)r * sub.size + (w0 >> 16)) * MG + g] += v;
            }
            const int cnt = *sh.cnt;
            __syncthreads();
            if (cnt > list_cap - S::TERMS * PT) near_flush<MG, EV>(P, sub, sub_tets, i0, g0, sh);
        }
    }
    near_flush<MG, EV>(P, sub, sub_tets, i0, g0, sh);
}

// The gather lists of one pass: its tetrahedra's vertices inside the sub-cluster,
// sorted by column (then by position), as offsets into the stage.
template <int MG, int EV>
__global__ void __launch_bounds__(256) pass_lists_kernel(const int4* __restrict__ tet, const SubInfo* __restrict__ subs,
                                                         const int* __restrict__ pass_sub, const int* __restrict__ sub_tets,
                                                         int PT, uint16_t* __restrict__ ref, unsigned* __restrict__ run)
{
    using S = RowShape<MG, EV>;
    extern __shared__ short loc[];   // [4 PT]
    __shared__ int scan[2][256];
    const SubInfo sub = subs[pass_sub[blockIdx.x]];
    const int p = blockIdx.x - sub.pass0, j = threadIdx.x;
    const int nt = min(PT, sub.ntet - p * PT);
    uint16_t* pref = ref + (int64_t)blockIdx.x * 4 * PT;
    unsigned* prun = run + (int64_t)blockIdx.x * kRunWords;
    for (int t = j; t < nt; t += 256) {
        const int4 tv = tet[sub_tets[sub.tet0 + p * PT + t]];
        const int id[4] = {tv.x, tv.y, tv.z, tv.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
            loc[4 * t + k] = (unsigned)(id[k] - sub.start) < (unsigned)sub.size ? (short)(id[k] - sub.start) : (short)-1;
    }
    __syncthreads();
    int n = 0;
    for (int e = 0; e < 4 * nt; ++e) n += loc[e] == j;
    scan[0][j] = n;
    scan[1][j] = n > 0;
    __syncthreads();
    for (int o = 1; o < 256; o <<= 1) {
        const int a = j >= o ? scan[0][j - o] : 0, b = j >= o ? scan[1][j - o] : 0;
        __syncthreads();
        scan[0][j] += a;
        scan[1][j] += b;
        __syncthreads();
    }
    int at = scan[0][j] - n;
    if (n > 0) prun[1 + scan[1][j] - 1] = ((unsigned)j << 16) | (unsigned)at;
    if (j == 255) {
        prun[0] = (unsigned)scan[1][255];
        prun[1 + scan[1][255]] = (unsigned)scan[0][255];
    }
    for (int e = 0; e < 4 * nt; ++e)
        if (loc[e] == j) pref[at++] = (uint16_t)((e >> 2) * S::RS + (e & 3) * MG);
}

// ---- pivot columns ---------------------------------------------------------------
// Column j for rows row0 .. row0 + m - 1, at most one row per thread a call: with
// fewer rows, several threads share a row's tetrahedra.  The column's points are
// the same for every row: a batch of kColTets tetrahedra is staged in shared
// memory, and a warp's lanes read one point together.
constexpr int kColTets = 32;
template <int MG>
struct ColShared {
    float4 pt[kColTets][4], cs[kColTets][4];
    float4 cen[kColTets];
    int tet[kColTets];
    float red[1];   // [threads][MG], past the end of the struct
    static constexpr int bytes(int nt) { return (int)sizeof(ColShared) + 4 * MG * nt; }
};

// out[g * gstride + row]: the finished sums times c_g, rows r0 .. r0 + mc - 1 (mc <= threads)
template <int MG, int EV>
__device__ __forceinline__ void column_chunk(const KernelParams& P, int row0, int mc, int j, int g0, ColShared<MG>& sh,
                                             float* __restrict__ out, int64_t gstride, unsigned& n_terms, unsigned& n_depths)
{
    const int tid = threadIdx.x, nth = blockDim.x;
    const int parts = nth / mc;
    const int part = tid / mc, pos = tid - part * mc;
    const bool live = part < parts;
    const int i = row0 + (live ? pos : 0);
    const Vec3<float> xi = load_xyz<float>(P, i);
    GroupSum<MG> acc;
    acc.zero();
    const int t0 = P.vt_ptr[j], t1 = P.vt_ptr[j + 1];
    for (int b0 = t0; b0 < t1; b0 += kColTets) {
        const int nt = min(kColTets, t1 - b0);
        __syncthreads();   // the previous batch is no longer read
        for (int e = tid; e < nt * 4; e += nth) {
            const int t = e >> 2, q = e & 3;
            const int packed = P.vt_idx[b0 + t], tet = packed >> 2;
            float4 y4 = P.tpt[(int64_t)q * P.T + tet];
            y4.w *= q == (packed & 3) ? kTetB + kTetG : kTetB;
            sh.pt[t][q] = y4;
            if constexpr (EV == EV_PHASE) {
                if (P.sinprod) sh.cs[t][q] = P.tcos[(int64_t)q * P.T + tet];
            }
            if (q == 0) {
                sh.cen[t] = P.tcen[tet];
                sh.tet[t] = packed;
            }
        }
        __syncthreads();
        if (!live) continue;
        unsigned near[EV == EV_PHASE ? 2 : 1];   // near tetrahedra of this row: direct, reflected term
        near[0] = 0u;
        if constexpr (EV == EV_PHASE) {
            near[1] = 0u;
            const PhasePoint x = phase_point(P, i);
            const Vec3<float> xb = P.has_wall ? mirror_point<float>(P, xi) : xi;
#pragma unroll 1
            for (int t = part; t < nt; t += parts) {
                const float4 c4 = sh.cen[t];
                const Vec3<float> cen = {c4.x, c4.y, c4.z};
                const bool fd = !(dist2<float>(xi, cen) < c4.w);
                const bool fr = P.has_wall && !(dist2<float>(xb, cen) < c4.w);
                if (!fd) near[0] |= 1u << t;
                if (P.has_wall && !fr) near[1] |= 1u << t;
                n_terms += (fd ? 4 : 14) + (P.has_wall ? (fr ? 4 : 14) : 0);
                n_depths += (fd ? 4 : 14) + (P.has_wall ? 2 * (fr ? 4 : 14) : 0);
#pragma unroll 1
                for (int q = 0; q < 4; ++q) {
                    const float4 y4 = sh.pt[t][q], yc = sh.cs[t][q];
                    float w, tau;
                    if (fd) {
                        phase_direct(P, x, y4, yc, w, tau);
                        acc.add(P, g0, w, tau);
                    }
                    if (fr) {
                        phase_reflected(P, x, y4, yc, w, tau);
                        acc.add(P, g0, w, tau);
                    }
                }
            }
        }
        const int nt_terms = term_count<EV == EV_GENERAL>(P);
#pragma unroll 1
        for (int t = 0; t < nt_terms; ++t) {
            if (!term_present(P, t)) continue;
            Vec3<float> src;
            float scale;
            source_of<EV == EV_GENERAL>(P, t, xi, src, scale);
            unsigned todo;
            if constexpr (EV == EV_PHASE) todo = near[t];
            else todo = nt == 32 ? ~0u : (1u << nt) - 1u;
            while (todo) {
                const int k = __ffs(todo) - 1;
                todo &= todo - 1;
                if (EV != EV_PHASE && k % parts != part) continue;
                const int tet = sh.tet[k] >> 2, slot = sh.tet[k] & 3;
                bool nr = true;
                if constexpr (EV != EV_PHASE) {
                    const float4 c4 = sh.cen[k];
                    nr = dist2<float>(src, {c4.x, c4.y, c4.z}) < c4.w;
                    const int legs = t == 0 ? 1 : (t == 1 ? 2 : P.xkind[t - 2] + 1);
                    n_terms += nr ? 14 : 4;
                    n_depths += (nr ? 14 : 4) * legs;
                    if (!nr) {
#pragma unroll 1
                        for (int q = 0; q < 4; ++q) {
                            const float4 y4 = sh.pt[k][q];
                            float w, tau;
                            if (general_term<EV == EV_GENERAL>(P, t, xi, src, scale, {y4.x, y4.y, y4.z}, y4.w, w, tau)) acc.add(P, g0, w, tau);
                        }
                        continue;
                    }
                }
                const int4 tv = P.tet[tet];
                const Vec3<float> v[4] = {load_xyz<float>(P, tv.x), load_xyz<float>(P, tv.y), load_xyz<float>(P, tv.z),
                                          load_xyz<float>(P, tv.w)};
                const float vol = P.tvol32[tet];
#pragma unroll 1
                for (int q = 0; q < 14; ++q) {
                    Vec3<float> y;
                    float b[4], w, tau;
                    const float w0 = near_point<EV == EV_GENERAL>(P, v, vol, q, y, b);
                    const float lam = slot == 0 ? b[0] : (slot == 1 ? b[1] : (slot == 2 ? b[2] : b[3]));
                    if (general_term<EV == EV_GENERAL>(P, t, xi, src, scale, y, w0 * lam, w, tau)) acc.add(P, g0, w, tau);
                }
            }
        }
    }
    // parts of a row summed in order
    if (parts > 1) {
        __syncthreads();
        if (live) acc.store(sh.red + (part * mc + pos) * MG);
        __syncthreads();
        for (int e = tid; e < mc * MG; e += nth) {
            const int g = e / mc, r = e - g * mc;
            if (g0 + g >= P.G) break;
            float v = 0.f;
            for (int k = 0; k < parts; ++k) v += sh.red[(k * mc + r) * MG + g];
            out[(int64_t)(g0 + g) * gstride + r] = times_c(P, v, g0 + g);
        }
    } else if (live) {
#pragma unroll
        for (int g = 0; g < MG; ++g)
            if (g0 + g < P.G) out[(int64_t)(g0 + g) * gstride + pos] = times_c(P, acc.get(g), g0 + g);
    }
    __syncthreads();
}

}  // namespace rt
