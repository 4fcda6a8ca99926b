#include "gemm_tile.h"

#include <algorithm>
#include <cmath>

namespace tn {

GemmForm gemm_form(const GemmShape& s, int sm_count) {
  GemmForm f;
  f.M = s.M;
  f.N = s.N;
  f.PA = s.PA;
  f.PB = s.PB;
  f.PC = s.PC;
  f.mapA_mode = s.mapA_mode;
  f.mapB_mode = s.mapB_mode;
  int cap = 16;
  while (cap < 256 && cap < s.tile_cap) cap *= 2;
  // Every pattern has its own A and all share B: one GEMM over the PC x M rows,
  // which lie one after another in A's planes and in C.  Small M then fills the
  // 128-row tiles, and a wave's row tiles share each B tile.
  if (f.mapA_mode == 0 && f.mapB_mode == 1 && f.PA == f.PC && f.PC > 1 && f.PC * f.M <= 0x7fffffffLL) {
    f.M *= f.PC;
    f.PA = f.PC = 1;
    f.mapA_mode = 1;
  }
  // All patterns share A and each has its own narrow B: the prepared B is one
  // matrix of all their columns, so this is one GEMM over PC x N columns whose
  // results go to their patterns.  53 patterns of one column each (2^18 x 2^6)
  // took 2.4 ms as 53 passes over A.
  if (f.mapA_mode == 1 && f.mapB_mode == 0 && f.PB == f.PC && f.PC > 1 && 2 * f.N < 16 &&
      f.PC * f.N <= 0x3fffffffLL && cap == 256) {
    f.sub_log2 = f.N == 1 ? 1 : f.N == 2 ? 2 : 3;
    f.N *= f.PC;
    f.PB = f.PC = 1;
    f.mapB_mode = 1;
  }
  // Tile width: the smallest of 16..cap that covers 2N, or, when all patterns
  // share A and 2N >= 16, up to cap columns of consecutive patterns folded side
  // by side (fold = BN / 2N, as many as the pattern count rounded up to a power
  // of two allows).  With a table of the patterns that read one A pattern, and
  // the widest tiles allowed, a tile takes the columns of one group of it.
  const int64_t N2 = 2 * f.N;
  int64_t w = N2;
  f.groups = f.PC;
  f.grouped = s.grp_fold > 0 && f.mapA_mode == 2 && cap == 256;
  if (f.grouped) {
    f.fold = s.grp_fold;
    w = N2 * f.fold;
    f.groups = s.n_groups;
  } else if (f.mapA_mode == 1 && f.PC > 1 && N2 >= 16 && N2 < cap) {
    while (w < cap && f.fold < f.PC) {
      w *= 2;
      f.fold *= 2;
    }
    f.groups = (f.PC + f.fold - 1) / f.fold;
  }
  while (f.bn < cap && f.bn < w) f.bn *= 2;
  // 256-wide tiles with at least 256 rows run on CTA pairs unless pair < 0.  In
  // tf32 a 128 x 256 tile on one CTA already feeds the tensor cores; pairs load
  // a third less per tile from L2, which is what bounds short K, and pay once
  // there are tiles for every pair: 53-qubit lattice in 3xTF32 23.3 -> 21.4 ms.
  f.paired = f.bn == 256 && f.M >= 2 * kGemmRows && s.pair >= 0;
  if (f.paired && s.h16 == 0) {
    const int64_t tiles =
        f.groups * ((f.M + 2 * kGemmRows - 1) / (2 * kGemmRows)) * (f.fold > 1 ? 1 : (N2 + 255) / 256);
    f.paired = tiles >= sm_count / 2;
  }
  return f;
}

// To set against the direct form's time (plan_direct).  Measured on GB300: about
// 4 us per launch; the passes stream at 5 TB/s and a GEMM writes C at 3.7 TB/s;
// it runs its tiles of 128 rows x BN real columns in whole waves of 152, each SM
// at its share of 280 (3xTF32) or 560 (16-bit) TFLOP/s for BN = 256, where an
// MMA narrower than 128 columns takes as long as one of 128.  The tiles are those
// of the launch: merged rows, joined columns and grouped patterns.  (Grouped ones
// priced pattern by pattern kept 32 patterns of 2^8 x 2^4 x 2^9 on the GEMM, whose
// 14 wide tiles take 41 us in one wave and 55 us with the preparations; the direct
// form takes 25 us.)
double tc_seconds(const GemmForm& f, int nk, double a, double b, double c, bool h16) {
  const double tiles = (double)f.groups * (f.fold > 1 ? 1.0 : std::ceil(2.0 * (double)f.N / f.bn)) *
                       std::ceil((double)f.M / kGemmRows);
  const double peak = h16 ? 560e12 : 280e12;
  const double tile_flops = 8.0 * kGemmRows * std::max(f.bn, 128) / 2.0 * std::ldexp(1.0, nk);
  const double mma = std::ceil(tiles / kGemmSMs) * tile_flops * kGemmSMs / peak;
  const double plane = h16 ? 8.0 : 16.0;
  const double gemm = std::max(mma, plane * a / 5.0e12 + 8.0 * c / 3.7e12);
  return gemm + (8.0 + plane) * a / 5.0e12 + (8.0 + 2.0 * plane) * b / 5.0e12 + 12e-6;
}

}  // namespace tn
