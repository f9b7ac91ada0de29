// rt_rows.h -- host side of the FP32 row and column evaluation: work items and
// one RowEval per evaluator, each compiled in its own translation unit
// (rt_rows_phase.cu, rt_rows_plain.cu, rt_rows_general.cu) so that the
// instances compile in parallel.
#pragma once

#include "rt_internal.h"

namespace rt {

// ACA rows (mode 0) / columns (mode 1) of the active far blocks.
struct AcaActive {
    int b;          // far block id
    int row0, m, col0, n;
    int64_t rbuf;   // offset of this block's [G][n] row buffer
    int64_t cbuf;   // offset of this block's [G][m] column buffer
    int64_t first_row, first_col;   // prefix of n (rows) and m (cols) over the active list
    int64_t uoff, voff;             // pool offsets of this step's u [G][m] and v [G][n]
    int64_t dot0;                   // first entry of this block's rank+1 dot products this step
    int64_t first_chunk;            // prefix of ceil(m / kColRows) over the active list
    int skip;       // set by the pivot kernel: zero row, no rank this step
};


// Row segments: rows i .. i + nrow - 1 over one sub-cluster of columns.
struct RowItem {
    int b;            // ACA block (row = i + istar[b]) or -1 (rows i ...)
    int i, nrow;
    int sub;
    int64_t out;      // output offset of (first row, first column, group 0); rows are adjacent
    int64_t gs, js;   // group and column strides of the output
};

// A sub-cluster: columns [start, start + size) and its tetrahedra
struct SubInfo {
    int start, size, tet0, ntet, pass0;
};

// threads of a pivot-column CTA; the chunks of a block's rows are of equal size
constexpr int kColThreads = 128;
__host__ __device__ inline int col_chunks(int m) { return (m + kColThreads - 1) / kColThreads; }

// Groups per chunk of the row and column kernels.  The phase evaluator's terms
// cost about as much as 16 groups' exponentials and sums, and its chunks of 16
// keep four CTAs on an SM; the others' terms cost several times that, so they
// take up to 32 groups at once.
inline int group_chunk(const Operator& op)
{
    const int G = op.G;
    return G <= 1 ? 1 : (G <= 4 ? 4 : (G <= 8 ? 8 : (G <= 16 || op.kp.evaluator == EV_PHASE ? 16 : 32)));
}

template <int EV>
struct RowEval {
    // device tables (sub-clusters, gather lists, point tables) for the sub-clusters' tetrahedra
    static int tables(Operator& op, const std::vector<int>& tets, std::string& err);
    // rows of device items; sums: most (rows x columns) of one item
    static int rows(Operator& op, const RowItem* items, int n, int sums, const int* istar, float* out, cudaStream_t s,
                    std::string& err);
    // pivot columns of the active blocks
    static int columns(Operator& op, const AcaActive* act, int na, int64_t nchunks, const int* jstar, float* out,
                       cudaStream_t s, std::string& err);
};

// CALL with EV the operator's evaluator
#define RT_EVALUATOR(op, CALL)                            \
    ((op).kp.evaluator == EV_PHASE     ? RowEval<EV_PHASE>::CALL   \
     : (op).kp.evaluator == EV_PLAIN   ? RowEval<EV_PLAIN>::CALL   \
                                       : RowEval<EV_GENERAL>::CALL)

}  // namespace rt
