// rt_pool.h -- capacity of the ACA term pool (host code without CUDA, so that
// it can be checked on its own).
#pragma once

#include <algorithm>
#include <cstdint>

namespace rt {

// Floats.  A wave's pool starts with room for kPoolTerms terms a block and, when
// it runs out, is replaced by a larger one whose new terms start where the old
// one ended.  Terms are whole float4s (aca_term_size) and are read and written as
// such, so every capacity has to be a multiple of 4: growth by half alone leaves
// that after a few steps (24 S, 36 S, 54 S, 81 S, 121.5 S for terms of S floats).
constexpr int64_t kPoolTerms = 24;
constexpr int64_t kPoolAlign = 64;
constexpr int64_t pool_round(int64_t n) { return (n + kPoolAlign - 1) / kPoolAlign * kPoolAlign; }

// the first pool of a wave whose blocks take `need` floats for a term each
constexpr int64_t pool_first(int64_t need) { return pool_round(kPoolTerms * need); }
// the pool after one of cap floats, when the blocks still active take `need` floats for a term each
constexpr int64_t pool_grown(int64_t cap, int64_t need) { return pool_round(std::max(cap + cap / 2, cap + 8 * need)); }

}  // namespace rt
