// rt_rows.h -- host side of the FP32 row and column evaluation: work items and
// one RowEval per evaluator, each compiled in its own translation unit
// (rt_rows_phase.cu, rt_rows_plain.cu, rt_rows_general.cu) so that the
// instances compile in parallel.
#pragma once

#include <algorithm>

#include "rt_internal.h"

namespace rt {

// State of a wave of admissible blocks during ACA (rt_aca.cuh); block b of the
// wave.  A term of block b: u [G][m4] then v [G][n4] at toff[b][l] of the pool,
// rows padded with zeros to multiples of four for 16-byte loads (a term's offset
// is a multiple of four too: rt_pool.h).
__host__ __device__ inline int round4(int x) { return (x + 3) & ~3; }
inline int64_t aca_term_size(int G, int m, int n) { return (int64_t)G * (round4(m) + round4(n)); }
enum { ACA_ACTIVE = 0, ACA_DONE = 1, ACA_DENSE = 2 };
struct AcaDev {
    int G, rmax, nb;
    double eps;
    const FarBlock* blk;
    const int *sub_ptr, *sub_of;   // sub-clusters of every cluster
    const int* order;   // [nb] largest blocks first
    int* next;          // next entry of order to take
    int* max_steps;
    int *istar, *rank, *steps, *status;
    double* norm2;      // [nb][G]
    float* wscale;      // [nb][G]   score weights 1/w_g
    int64_t* toff;      // [nb][rmax]
    unsigned char* used;   // [sum m]
    int64_t* used_off;  // [nb]
    float* pool;
    int64_t pool_cap;   // elements
    unsigned long long* pool_used;
};

// Row segments: rows i .. i + nrow - 1 over one sub-cluster of columns.
struct RowItem {
    int i, nrow;
    int sub;
    int64_t out;      // output offset of (first row, first column, group 0); rows are adjacent
    int64_t gs, js;   // group and column strides of the output
};

// A sub-cluster: columns [start, start + size) and its tetrahedra
struct SubInfo {
    int start, size, tet0, ntet, pass0;
};

// Groups per chunk of the row and column kernels.  The phase evaluator's terms
// cost about as much as 16 groups' exponentials and sums, and its chunks of 16
// keep four CTAs on an SM; the others' terms cost several times that, so they
// take up to 32 groups at once.
inline int group_chunk(int G, int ev)
{
    return G <= 1 ? 1 : (G <= 4 ? 4 : (G <= 8 ? 8 : (G <= 16 || ev == EV_PHASE ? 16 : 32)));
}
inline int group_chunk(const Operator& op) { return group_chunk(op.G, op.kp.evaluator); }

// Threads of a row or ACA CTA.  One CTA runs a block's whole ACA: with few
// admissible blocks more threads share a block, and with many, 128-thread CTAs
// waste the least on a block's ragged sizes.  Measured builds (near + ACA, ms) at
// 128 | 256 | 512 threads: phase evaluator 28 blocks 2.6 | 1.7 | 1.5, 334 blocks 3.8 |
// 2.5 | 2.7, 1818 blocks 8.0 | 6.0 | 9.0, 2970 blocks 19.1 | 15.0 | 22.2 (2 groups) and
// 28.8 | 29.7 | 36.1 (5 groups), 8466 blocks 65 | 73 | 90; general evaluator 298
// blocks 431 | 379 | 194; plain 1826 blocks 12.5 | 11.2 | 13.3.  A chunk of 32 groups
// needs 255 registers, so its CTAs stay at 256 threads.
inline int eval_threads(int G, int ev, size_t nb)
{
    if (group_chunk(G, ev) > 16) return nb < 608 ? 256 : 128;
    if (nb < (ev == EV_PHASE ? 320 : 608)) return 512;
    return nb < 3000 ? 256 : 128;
}
inline int eval_threads(const Operator& op) { return eval_threads(op.G, op.kp.evaluator, op.plan.far_blocks.size()); }

constexpr int kRunWords = kSubCols + 4;   // per pass: run count, runs, end mark
constexpr int tets_per_thread(int mg, int ev) { return mg == 1 && ev == EV_PHASE ? 4 : 1; }

// rows of one near-block item: the more, the wider the stores of a column's rows; the
// sums of all its rows take at most 8 KB, which keeps four CTAs on an SM at 16 groups
inline int rows_per_item(int mg, int n) { return std::max(1, std::min(8, 8192 / (4 * mg * n))); }

// Device bytes of the tables and near-block items that live until the near blocks are
// done (RowEval::tables, launch_rows), before anything is built: a sub-cluster of k
// vertices touches at most the sum of its vertices' tetrahedra (about half of it on a
// Kuhn mesh, whose tetrahedra share vertices).
int64_t eval_bytes_bound(const Plan& P, int64_t T, int G, int ev);

template <int EV>
struct RowEval {
    // what this unit needs once per device: its quadrature rules, its kernels' shared memory
    static int setup(std::string& err);
    // device tables (sub-clusters, gather lists, point tables) for the sub-clusters' tetrahedra
    static int tables(Operator& op, const std::vector<int>& tets, std::string& err);
    // rows of device items; sums: most (rows x columns) of one item
    static int rows(Operator& op, const RowItem* items, int n, int sums, float* out, cudaStream_t s, std::string& err);
    // ACA of the wave's active blocks, as far as the pool reaches; sums: columns of
    // the widest sub-cluster
    static int aca(Operator& op, const AcaDev& D, int sums, cudaStream_t s, std::string& err);
};

// CALL with EV the operator's evaluator
#define RT_EVALUATOR(op, CALL)                            \
    ((op).kp.evaluator == EV_PHASE     ? RowEval<EV_PHASE>::CALL   \
     : (op).kp.evaluator == EV_PLAIN   ? RowEval<EV_PLAIN>::CALL   \
                                       : RowEval<EV_GENERAL>::CALL)

}  // namespace rt
