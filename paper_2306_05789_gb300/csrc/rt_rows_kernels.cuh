// rt_rows_kernels.cuh -- kernels over row items and pivot columns, and the host
// side of one evaluator (RowEval<EV>, rt_rows.h).
#pragma once

#include <algorithm>
#include <mutex>

#include "rt_aca.cuh"

namespace rt {

template <int MG, int EV>
__global__ void __launch_bounds__(max_threads(MG, EV), 1) row_items_kernel(KernelParams P, const RowItem* __restrict__ items,
                                                                   const SubInfo* __restrict__ subs,
                                                                   const int* __restrict__ sub_tets,
                                                                   const uint16_t* __restrict__ pass_ref,
                                                                   const unsigned* __restrict__ pass_run,
                                                                   float* __restrict__ out)
{
    extern __shared__ __align__(16) char smem[];
    __shared__ int cnt;
    const RowItem it = items[blockIdx.x];
    const SubInfo sub = subs[it.sub];
    const int g0 = blockIdx.y * MG, ng = min(MG, P.G - g0), n = sub.size;
    const RowShared<MG, EV> sh(smem, &cnt);
    unsigned n_terms = 0, n_depths = 0;
    row_segment<MG, EV>(P, sub, sub_tets, pass_ref, pass_run, it.i, it.nrow, g0, sh, n_terms, n_depths);
    if (g0 == 0) count_work(P, n_terms, n_depths);
    const int per = it.nrow * n;
    for (int e = threadIdx.x; e < per * ng; e += blockDim.x) {
        const int g = e / per, k = e - g * per;
        const int j = k / it.nrow, r = k - j * it.nrow;
        out[it.out + r + (int64_t)(g0 + g) * it.gs + (int64_t)j * it.js] = times_c(P, sh.acc[((int64_t)r * n + j) * MG + g], g0 + g);
    }
}

// MACRO(MG, EV) for the operator's chunk width
#define RT_DISPATCH_MG(op, MACRO)                         \
    do {                                                  \
        const int mg_ = group_chunk(op);                  \
        if (mg_ == 1) MACRO(1, EV);                       \
        else if (mg_ == 4) MACRO(4, EV);                  \
        else if (mg_ == 8) MACRO(8, EV);                  \
        else if (mg_ == 16) MACRO(16, EV);                \
        else if constexpr (EV != EV_PHASE) MACRO(32, EV); \
    } while (0)

template <int EV>
int RowEval<EV>::setup(std::string& err)
{
    const int rc = upload_rules(err);
    if (rc) return rc;
    static bool attr_set[64] = {false};
    static std::mutex mu;
    std::lock_guard<std::mutex> lock(mu);
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 64 && !attr_set[dev]) {
#define RT_ROW_ATTR(MG, EV) \
    RT_CUDA_TRY(cudaFuncSetAttribute(row_items_kernel<MG, EV>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024)); \
    RT_CUDA_TRY(cudaFuncSetAttribute(aca_block_kernel<MG, EV>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024))
        RT_ROW_ATTR(1, EV);
        RT_ROW_ATTR(4, EV);
        RT_ROW_ATTR(8, EV);
        RT_ROW_ATTR(16, EV);
        if constexpr (EV != EV_PHASE) {
            RT_ROW_ATTR(32, EV);
        }
#undef RT_ROW_ATTR
        attr_set[dev] = true;
    }
    return RT_OK;
}

// Device tables of the row and column evaluation: sub-clusters, gather lists,
// point tables (rt_rows.cuh, rt_phase.cuh).  They live until the assembly ends.
template <class T>
static int table_alloc(Operator& op, T** p, size_t count, std::string& err)
{
    *p = nullptr;
    const cudaError_t e = cudaMallocAsync((void**)p, std::max<size_t>(count, 1) * sizeof(T), op.stream);
    if (e != cudaSuccess) {
        *p = nullptr;
        err = std::string("cudaMallocAsync (assembly tables): ") + cudaGetErrorString(e);
        return RT_ENOMEM;
    }
    op.eval_tables.push_back((void*)*p);
    op.eval_bytes += (int64_t)(count * sizeof(T));
    return RT_OK;
}

template <int EV>
int RowEval<EV>::tables(Operator& op, const std::vector<int>& tets, std::string& err)
{
    int rc;
    cudaStream_t s = op.stream;
    int pt = 0;
    const int nth = eval_threads(op);
#define RT_PASS_TETS(MG, EV) pt = RowShape<MG, EV>::TPT * nth
    RT_DISPATCH_MG(op, RT_PASS_TETS);
#undef RT_PASS_TETS
    const int nsub = (int)op.sub_start.size();
    std::vector<SubInfo> subs(nsub);
    std::vector<int> pass_sub;
    for (int k = 0; k < nsub; ++k) {
        const int t0 = op.sub_tet_ptr[k], nt = op.sub_tet_ptr[k + 1] - t0;
        subs[k] = {op.sub_start[k], op.sub_size[k], t0, nt, (int)pass_sub.size()};
        pass_sub.insert(pass_sub.end(), (nt + pt - 1) / pt, k);
    }
    const size_t np = pass_sub.size();
    SubInfo* d_subs;
    int* d_pass_sub;
    if ((rc = table_alloc(op, &op.d_sub_tets, tets.size(), err))) return rc;
    if ((rc = table_alloc(op, &d_subs, subs.size(), err))) return rc;
    if ((rc = table_alloc(op, &d_pass_sub, np, err))) return rc;
    if ((rc = table_alloc(op, &op.d_pass_ref, np * 4 * pt, err))) return rc;
    if ((rc = table_alloc(op, &op.d_pass_run, np * kRunWords, err))) return rc;
    if ((rc = upload_async(op, op.d_sub_tets, tets.data(), tets.size(), err))) return rc;
    if ((rc = upload_async(op, d_subs, subs.data(), subs.size(), err))) return rc;
    if ((rc = upload_async(op, d_pass_sub, pass_sub.data(), np, err))) return rc;
    op.d_subs = d_subs;
    float4 *cen, *pts, *cs = nullptr, *px = nullptr, *pc = nullptr;
    if ((rc = table_alloc(op, &cen, op.T, err))) return rc;
    if ((rc = table_alloc(op, &pts, (size_t)4 * op.T, err))) return rc;
    if constexpr (EV == EV_PHASE) {
        if ((rc = table_alloc(op, &cs, op.kp.sinprod ? (size_t)4 * op.T : 1, err))) return rc;
        if ((rc = table_alloc(op, &px, op.N, err))) return rc;
        if ((rc = table_alloc(op, &pc, op.N, err))) return rc;
        phase_vertex_table<<<(op.N + 255) / 256, 256, 0, s>>>(op.kp, px, pc);
        tet_point_table<true, false><<<(op.T + 127) / 128, 128, 0, s>>>(op.kp, cen, pts, cs);
    } else {
        tet_point_table<false, EV == EV_GENERAL><<<(op.T + 127) / 128, 128, 0, s>>>(op.kp, cen, pts, nullptr);
    }
    op.kp.pxyz = px;
    op.kp.pcos = pc;
    op.kp.tcen = cen;
    op.kp.tpt = pts;
    op.kp.tcos = cs;
    if (np > 0) {
#define RT_PASS_LISTS(MG, EV) \
    pass_lists_kernel<MG, EV><<<(unsigned)np, 256, 4 * pt * sizeof(short), s>>>(op.d_tet, d_subs, d_pass_sub,       \
                                                                                op.d_sub_tets, pt, op.d_pass_ref, \
                                                                                op.d_pass_run)
        RT_DISPATCH_MG(op, RT_PASS_LISTS);
#undef RT_PASS_LISTS
    }
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
}

template <int EV>
int RowEval<EV>::rows(Operator& op, const RowItem* items, int n, int sums, float* out, cudaStream_t s, std::string& err)
{
    const int mg = group_chunk(op), nth = eval_threads(op);
    const dim3 grid((unsigned)n, (op.G + mg - 1) / mg);
#define RT_LAUNCH_ROWS(MG, EV)                                                                                  \
    row_items_kernel<MG, EV><<<grid, nth, RowShape<MG, EV>::fixed(nth) + (size_t)sums * MG * sizeof(float), \
                               s>>>(op.kp, items, (const SubInfo*)op.d_subs, op.d_sub_tets, op.d_pass_ref,      \
                                    op.d_pass_run, out)
    RT_DISPATCH_MG(op, RT_LAUNCH_ROWS);
#undef RT_LAUNCH_ROWS
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
}

template <int EV>
int RowEval<EV>::aca(Operator& op, const AcaDev& D, int sums, cudaStream_t s, std::string& err)
{
    const int nth = eval_threads(op);
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, op.device);
#define RT_LAUNCH_ACA(MG, EV)                                                                                         \
    do {                                                                                                              \
        const size_t bytes = aca_phase_bytes<MG, EV>(nth) + (size_t)sums * MG * sizeof(float);                           \
        int per_sm = 1;                                                                                               \
        RT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, aca_block_kernel<MG, EV>, nth, bytes)); \
        const int grid = std::max(1, std::min(D.nb, std::max(1, per_sm) * sms));                                      \
        aca_block_kernel<MG, EV><<<grid, nth, bytes, s>>>(op.kp, D, (const SubInfo*)op.d_subs, op.d_sub_tets, \
                                                                  op.d_pass_ref, op.d_pass_run);                      \
    } while (0)
    RT_DISPATCH_MG(op, RT_LAUNCH_ACA);
#undef RT_LAUNCH_ACA
    RT_CUDA_TRY(cudaGetLastError());
    return RT_OK;
}

}  // namespace rt
