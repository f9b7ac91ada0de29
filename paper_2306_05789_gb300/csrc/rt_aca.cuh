// rt_aca.cuh -- partially pivoted ACA of the admissible blocks (Section 2.1),
// pivots shared by all groups, one CTA per block from the first pivot row to
// the stopping test.
//
// Every admissible block b (m x n) is approximated for all groups g at once:
//   step k: residual row  R_g = G_g[i*, :] - sum_{l<k} u_{g,l}[i*] v_{g,l}
//           pivot column  j*  = argmax_j sum_g |R_g[j]| / w_g   (first index on ties)
//           v_g = R_g / R_g[j*]           (skipped for a group whose pivot is 0)
//           u_g = G_g[:, j*] - sum_{l<k} u_{g,l} v_{g,l}[j*]
//           ||S_g||_F^2 += 2 sum_{l<k} (u_l.u)(v_l.v) + |u|^2 |v|^2      (FP64)
//           group g done when |u_g| |v_g| <= eps ||S_g||_F
//           next row i* = argmax over unused rows of sum_g |u_g[i]| / w_g
// w_g = ||S_g||_F (1 before the first term) puts the groups on one scale.
// A block stops when every group is done; when another term would make
// r (m + n) >= m n, or the rank limit is reached, it is stored dense.
// The first pivot row is the block's first row.
//
// Blocks are independent, so a CTA takes one from a list (largest first) and
// runs all its steps: no launches, copies or host waits between the steps, and
// the panels of the few hundred blocks in flight stay in L2 for the residuals
// and norm updates, which read every earlier term twice a step.  (Launched
// step by step over all blocks, those passes went to HBM: 135 of 300 ms at
// 32^3 with 16 groups, and every step waited for the host and for its slowest
// block.)  Terms come from a pool through one atomic offset; a block that finds
// it empty leaves its state and a later launch, with a larger pool, resumes it.
// Bound: instruction issue of the row and column evaluation.
// Measured on GB300, the whole ACA of one operator, before (one launch per
// phase and step) and after: 32^3 x 16 groups 330 -> 248 ms, 41^3 x 1 group 386 ->
// 291 ms, 13^3 x 3 groups 9.7 -> 6.0 ms (4.0 ms with 256 threads, eval_threads).  Six CTAs an SM and loops that are not
// unrolled over the points matter: at four CTAs and unrolled, 431 ms at 41^3,
// with the warps waiting for instructions (2.6 of 7.4 stall cycles an issue).
#pragma once

#include "rt_rows.cuh"

namespace rt {

__device__ __forceinline__ unsigned long long score_key(float s, int idx)
{
    if (!(s >= 0.0f) || isinf(s)) s = 0.0f;
    return ((unsigned long long)__float_as_uint(s) << 32) | (unsigned long long)(0xffffffffu - (unsigned)idx);
}

constexpr int kAcaWarps = 24;    // most warps of a CTA
constexpr int kNormWarps = 8;    // most warps of the norm update
constexpr int kCoefs = 1024;     // coefficients of one chunk of earlier terms
constexpr int kTermChunk = 64;   // most earlier terms per chunk

// Scratch of the residual and norm phases; shares its memory with the row and
// column evaluation's (except the row sums).
struct AcaScratch {
    double cross[kNormWarps][kMaxGroups], uu[kMaxGroups], vv[kMaxGroups];
    int64_t off[kTermChunk];
    float coef[kCoefs];
};

// State of the CTA's block that outlives a phase.
struct AcaState {
    double norm2[kMaxGroups];
    float ws[kMaxGroups], inv[kMaxGroups];
    unsigned rowmax[kMaxGroups];
    unsigned long long key[kAcaWarps];
    int64_t slot;
    int item, next;
};

// bytes shared by all phases of nt threads (without the row sums), 16-byte multiple
template <int MG, int EV>
__host__ __device__ constexpr int aca_phase_bytes(int nt)
{
    int b = RowShape<MG, EV>::fixed(nt);
    b = b > ColShared<MG>::bytes(nt) ? b : ColShared<MG>::bytes(nt);
    b = b > (int)sizeof(AcaScratch) ? b : (int)sizeof(AcaScratch);
    return (b + 15) & ~15;
}

__device__ __forceinline__ unsigned long long block_max(unsigned long long k, unsigned long long (&s)[kAcaWarps])
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, k, o);
        k = v > k ? v : k;
    }
    __syncthreads();   // the previous maximum has been read
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = k;
    __syncthreads();
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) k = s[w] > k ? s[w] : k;
    return k;
}

// buf[g][e] -= sum_{l<r} c_{l,g} panel_l[g][e], e < ld: c_{l,g} = other_l[g][idx].
// Panels of term l start at toff[l] + own (rows of ld), the other side's at
// toff[l] + oth (rows of old).  Bound by L2 latency: 16-byte loads, eight terms
// in flight per thread.
static __device__ __noinline__ void aca_residual(float* pool, const int64_t* toff, int r, int G, int64_t own, int ld, int64_t oth,
                                          int old, int idx, float* buf, AcaScratch& sc)
{
    const int tid = threadIdx.x, nth = blockDim.x, ld4 = ld >> 2;
    const int lc_max = min(kTermChunk, kCoefs / G);
    for (int l0 = 0; l0 < r; l0 += lc_max) {
        const int lc = min(lc_max, r - l0);
        __syncthreads();
        if (tid < lc) sc.off[tid] = toff[l0 + tid] + own;
        for (int e = tid; e < lc * G; e += nth) {
            const int l = e / G, g = e - l * G;
            sc.coef[e] = pool[toff[l0 + l] + oth + (int64_t)g * old + idx];
        }
        __syncthreads();
        for (int k = tid; k < G * ld4; k += nth) {
            const int g = k / ld4;
            float4 x = reinterpret_cast<float4*>(buf)[k];
#pragma unroll 8
            for (int l = 0; l < lc; ++l) {
                const float c = sc.coef[l * G + g];
                const float4 p = reinterpret_cast<const float4*>(pool + sc.off[l])[k];
                x.x -= c * p.x;
                x.y -= c * p.y;
                x.z -= c * p.z;
                x.w -= c * p.w;
            }
            reinterpret_cast<float4*>(buf)[k] = x;
        }
    }
    __syncthreads();
}

// Norm update sums: (u_l.u) (v_l.v) of the earlier terms into sc.cross, |u|^2
// and |v|^2 of the new one.  A warp takes a term; its lanes are split among gp
// groups (L = 32 / gp >= 8 lanes a group): FP32 sums per lane, FP64 across lanes.
static __device__ __noinline__ void aca_norm_sums(const float* pool, const int64_t* toff, int64_t slot, int r, int G, int ldm, int ldn,
                                           AcaScratch& sc)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int gp = 1;
    while (gp < G && gp < 4) gp <<= 1;
    const int L = 32 / gp, sl = lane % L;
    const int64_t um = (int64_t)G * ldm;
    const float4 *nu = reinterpret_cast<const float4*>(pool + slot), *nv = reinterpret_cast<const float4*>(pool + slot + um);
    const int m4 = ldm >> 2, n4 = ldn >> 2;
    const int nw = min((int)(blockDim.x >> 5), kNormWarps);
    if (warp >= nw) return;
    for (int l = warp; l <= r; l += nw) {
        const int64_t at = l < r ? toff[l] : slot;
        const float4 *tu = reinterpret_cast<const float4*>(pool + at), *tv = reinterpret_cast<const float4*>(pool + at + um);
#pragma unroll 2
        for (int g0 = 0; g0 < G; g0 += gp) {
            const int g = g0 + lane / L;
            float pu = 0.f, pv = 0.f;
            if (g < G) {
                auto dot = [](const float4& a, const float4& b, float s) {
                    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, s))));
                };
#pragma unroll 4
                for (int i = sl; i < m4; i += L) pu = dot(tu[(int64_t)g * m4 + i], nu[(int64_t)g * m4 + i], pu);
#pragma unroll 4
                for (int j = sl; j < n4; j += L) pv = dot(tv[(int64_t)g * n4 + j], nv[(int64_t)g * n4 + j], pv);
            }
            double su = pu, sv = pv;
            for (int o = L >> 1; o > 0; o >>= 1) {
                su += __shfl_xor_sync(0xffffffffu, su, o);
                sv += __shfl_xor_sync(0xffffffffu, sv, o);
            }
            if (sl == 0 && g < G) {
                if (l < r) {
                    sc.cross[warp][g] += su * sv;
                } else {
                    sc.uu[g] = su;
                    sc.vv[g] = sv;
                }
            }
        }
    }
}

template <int MG, int EV>
__global__ void __launch_bounds__(max_threads(MG, EV), 1) aca_block_kernel(KernelParams P, AcaDev D,
                                                                                  const SubInfo* __restrict__ subs,
                                                                                  const int* __restrict__ sub_tets,
                                                                                  const uint16_t* __restrict__ pass_ref,
                                                                                  const unsigned* __restrict__ pass_run)
{
    extern __shared__ __align__(16) char smem[];
    __shared__ AcaState st;
    __shared__ int list_len;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nth = blockDim.x, G = D.G;
    RowShared<MG, EV> sh(smem, &list_len);
    sh.acc = (float*)(smem + aca_phase_bytes<MG, EV>(blockDim.x));
    ColShared<MG>& colsh = *reinterpret_cast<ColShared<MG>*>(smem);
    AcaScratch& sc = *reinterpret_cast<AcaScratch*>(smem);
    float* pool = D.pool;
    unsigned n_terms = 0, n_depths = 0;
    for (;;) {
        __syncthreads();
        if (tid == 0) st.item = atomicAdd(D.next, 1);
        __syncthreads();
        if (st.item >= D.nb) break;
        const int b = D.order[st.item];
        if (D.status[b] != ACA_ACTIVE) continue;
        const FarBlock fb = D.blk[b];
        const int m = fb.m, n = fb.n;
        const int ldm = round4(m), ldn = round4(n);
        const int64_t um = (int64_t)G * ldm;          // V starts here in a term
        const int64_t* toff = D.toff + (int64_t)b * D.rmax;
        unsigned char* used = D.used + D.used_off[b];
        int r = D.rank[b], is = D.istar[b], steps = D.steps[b], status = ACA_ACTIVE;
        if (tid < G) {
            st.norm2[tid] = D.norm2[(int64_t)b * G + tid];
            st.ws[tid] = D.wscale[(int64_t)b * G + tid];
        }
        bool have = false;
        while (status == ACA_ACTIVE) {
            if (steps >= D.rmax + 64) {
                status = ACA_DENSE;
                break;
            }
            if (!have) {
                if (tid == 0) {
                    const unsigned long long need = (unsigned long long)(um + (int64_t)G * ldn);
                    const unsigned long long at = atomicAdd(D.pool_used, need);
                    st.slot = at + need <= (unsigned long long)D.pool_cap ? (int64_t)at : -1;
                }
                __syncthreads();
                if (st.slot < 0) break;   // resumed by a later launch
                have = true;
                for (int k = tid; k < 4 * G; k += nth) {   // the rows' padding
                    const int g = k >> 2, o = k & 3;
                    if (m + o < ldm) pool[st.slot + (int64_t)g * ldm + m + o] = 0.f;
                    if (n + o < ldn) pool[st.slot + um + (int64_t)g * ldn + n + o] = 0.f;
                }
            }
            ++steps;
            float* u = pool + st.slot;
            float* v = u + um;
            // ---- pivot row
            for (int e = D.sub_ptr[fb.sc]; e < D.sub_ptr[fb.sc + 1]; ++e) {
                const SubInfo sub = subs[D.sub_of[e]];
                for (int g0 = 0; g0 < G; g0 += MG) {
                    unsigned nt = 0, nd = 0;
                    row_segment<MG, EV>(P, sub, sub_tets, pass_ref, pass_run, fb.row0 + is, 1, g0, sh, nt, nd);
                    if (g0 == 0) {
                        n_terms += nt;
                        n_depths += nd;
                    }
                    const int ng = min(MG, G - g0);
                    float* out = v + (int64_t)g0 * ldn + (sub.start - fb.col0);
                    for (int k = tid; k < ng * sub.size; k += nth) {
                        const int g = k / sub.size, j = k - g * sub.size;
                        out[(int64_t)g * ldn + j] = times_c(P, sh.acc[j * MG + g], g0 + g);
                    }
                    __syncthreads();
                }
            }
            aca_residual(pool, toff, r, G, um, ldn, 0, ldm, is, v, sc);
            // ---- pivot column: largest scaled residual; per group its largest value
            if (tid < G) st.rowmax[tid] = 0u;
            __syncthreads();
            unsigned long long key = 0ull;
            for (int j0 = warp * 32; j0 < n; j0 += nth) {
                const int j = j0 + lane;
                float score = 0.0f;
#pragma unroll 4
                for (int g = 0; g < G; ++g) {
                    const float x = j < n ? fabsf(v[(int64_t)g * ldn + j]) : 0.f;
                    score += x * st.ws[g];
                    const unsigned mx = __reduce_max_sync(0xffffffffu, isfinite(x) ? __float_as_uint(x) : 0u);
                    if (lane == 0 && mx) atomicMax(&st.rowmax[g], mx);
                }
                const unsigned long long k = j < n ? score_key(score, j) : 0ull;
                key = k > key ? k : key;
            }
            key = block_max(key, st.key);
            if (!(__uint_as_float((unsigned)(key >> 32)) > 0.0f)) {
                // exact zero row: mark it used and move to the first unused row
                if (tid == 0) {
                    used[is] = 1;
                    st.next = m;
                }
                __syncthreads();
                for (int i = tid; i < m; i += nth)
                    if (!used[i]) {
                        atomicMin(&st.next, i);
                        break;
                    }
                __syncthreads();
                if (st.next >= m) status = ACA_DONE;
                else is = st.next;
                __syncthreads();
                continue;
            }
            const int js = (int)(0xffffffffu - (unsigned)(key & 0xffffffffu));
            if (tid < G) {
                const float d = v[(int64_t)tid * ldn + js];
                // a group whose value at the shared pivot is negligible skips this term
                st.inv[tid] = (fabsf(d) > 1e-4f * __uint_as_float(st.rowmax[tid]) && fabsf(d) > 1e-37f) ? 1.0f / d : 0.0f;
            }
            // ---- pivot column of G, its residual, the next row
            {
                const int nch = (m + nth - 1) / nth, size = (m + nch - 1) / nch;   // chunks of equal size
                for (int r0 = 0; r0 < m; r0 += size)
                    for (int g0 = 0; g0 < G; g0 += MG) {
                        unsigned nt = 0, nd = 0;
                        column_chunk<MG, EV>(P, fb.row0 + r0, min(size, m - r0), fb.col0 + js, g0, colsh, u + r0, ldm, nt, nd);
                        if (g0 == 0) {
                            n_terms += nt;
                            n_depths += nd;
                        }
                    }
            }
            aca_residual(pool, toff, r, G, 0, ldm, um, ldn, js, u, sc);
            key = 0ull;
            for (int i = tid; i < m; i += nth) {
                float score = 0.0f;
#pragma unroll 4
                for (int g = 0; g < G; ++g) {
                    float x = u[(int64_t)g * ldm + i];
                    if (st.inv[g] == 0.0f) {
                        x = 0.0f;
                        u[(int64_t)g * ldm + i] = 0.0f;
                    }
                    score += fabsf(x) * st.ws[g];
                }
                if (i != is && !used[i]) {
                    const unsigned long long k = score_key(score, i);
                    key = k > key ? k : key;
                }
            }
            for (int k = tid; k < G * (ldn >> 2); k += nth) {
                const float inv = st.inv[k / (ldn >> 2)];
                float4 x = reinterpret_cast<float4*>(v)[k];
                x = make_float4(x.x * inv, x.y * inv, x.z * inv, x.w * inv);
                reinterpret_cast<float4*>(v)[k] = x;
            }
            for (int k = tid; k < kNormWarps * kMaxGroups; k += nth) (&sc.cross[0][0])[k] = 0.0;
            key = block_max(key, st.key);   // also orders the writes above
            aca_norm_sums(pool, toff, st.slot, r, G, ldm, ldn, sc);
            __syncthreads();
            bool done = true;
            if (tid < G) {
                double cross = 0.0;
#pragma unroll
                for (int w = 0; w < kNormWarps; ++w) cross += sc.cross[w][tid];
                const double q = sc.uu[tid] * sc.vv[tid];
                double s = st.norm2[tid] + 2.0 * cross + q;
                if (s < 0.0) s = 0.0;
                st.norm2[tid] = s;
                // a group that skipped this shared pivot (1/delta = 0) has learned nothing
                // from the term and is not declared converged by it
                done = st.inv[tid] != 0.0f && sqrt(q) <= D.eps * sqrt(s);
                st.ws[tid] = s > 0.0 ? (float)(1.0 / sqrt(s)) : 1.0f;
            }
            if (tid == 0) {
                D.toff[(int64_t)b * D.rmax + r] = st.slot;
                used[is] = 1;
            }
            const int all_done = __syncthreads_and(done ? 1 : 0);
            ++r;
            have = false;
            if (all_done) status = ACA_DONE;
            else if ((int64_t)(r + 1) * (m + n) >= (int64_t)m * n || r >= D.rmax) status = ACA_DENSE;
            else if (!(__uint_as_float((unsigned)(key >> 32)) > 0.0f))
                status = ACA_DONE;   // no unused row with a nonzero residual: exact on all rows seen
            else is = (int)(0xffffffffu - (unsigned)(key & 0xffffffffu));
        }
        __syncthreads();
        if (tid < G) {
            D.norm2[(int64_t)b * G + tid] = st.norm2[tid];
            D.wscale[(int64_t)b * G + tid] = st.ws[tid];
        }
        if (tid == 0) {
            D.rank[b] = r;
            D.istar[b] = is;
            D.steps[b] = steps;
            D.status[b] = status;
            atomicMax(D.max_steps, steps);
        }
    }
    count_work(P, n_terms, n_depths);
}

}  // namespace rt
