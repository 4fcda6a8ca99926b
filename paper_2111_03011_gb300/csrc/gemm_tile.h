// What a tensor-core GEMM (gemm_tc.cu) runs as: the merged shape, the tile and
// whether CTA pairs take it.  One rule for the dispatch, the tuner and the
// description of a plan.  Host-only, no CUDA headers.
#pragma once

#include <cstdint>

namespace tn {

constexpr int kGemmRows = 128;   // rows of a one-CTA tile; a CTA pair takes twice as many
constexpr int kGemmSMs = 152;    // of a GB300, where no device is asked

struct GemmShape {
  int64_t M = 1, N = 1;
  int64_t PA = 1, PB = 1, PC = 1;
  int mapA_mode = 1, mapB_mode = 1;   // 0 identity, 1 zero, 2 table
  int h16 = 0;                        // 0 tf32, 1 bf16, 2 fp16 operands
  int pair = 0;                       // -1: no CTA pairs
  int tile_cap = 256;                 // widest tile, real columns (16..256)
  int grp_fold = 0;                   // patterns per group where a table of pattern groups is given, else 0
  int64_t n_groups = 0;
};

struct GemmForm {
  int64_t M = 1, N = 1, PA = 1, PB = 1, PC = 1;   // after merging
  int mapA_mode = 1, mapB_mode = 1;
  int sub_log2 = -1;     // >= 0: the columns are many patterns', 2^sub_log2 reals each
  bool grouped = false;  // the table of pattern groups is used
  int bn = 16;           // real columns per tile: 16, 32, 64, 128 or 256
  int fold = 1;          // patterns side by side in a tile
  int64_t groups = 1;    // sets of patterns that tiles cover
  bool paired = false;   // 256 x 256 tiles on CTA pairs
};

GemmForm gemm_form(const GemmShape& s, int sm_count);

// Modelled time of a contraction that runs as f with 2^nk reductions: split
// permute, B preparation and tensor-core GEMM (a, b, c: elements of the
// operands and the result).
double tc_seconds(const GemmForm& f, int nk, double a, double b, double c, bool h16);

}  // namespace tn
