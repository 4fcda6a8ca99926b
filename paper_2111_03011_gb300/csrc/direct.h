// Direct contraction step (direct.cu): its launch parameters and how the tile,
// the roles of the operands and the split of K are chosen.  Host-only code is
// usable without CUDA headers (planner.cpp).
#pragma once

#include <cstdint>

namespace tn {

// Tile shapes: log2 of rows, columns and the k values per pipeline stage, and
// the rate the kernel reaches on it (complex multiply-adds per second of the
// padded tile, measured on long launches).
struct DirectConfig {
  int tr, tc, tk;
  double rate;
};
constexpr DirectConfig kDirectConfigs[] = {
    {6, 6, 4, 5.8e12}, {6, 5, 4, 5.0e12}, {6, 4, 5, 3.5e12}, {6, 2, 5, 1.7e12}, {6, 0, 5, 0.9e12},
    {4, 4, 6, 2.6e12}, {4, 2, 7, 2.0e12}, {4, 0, 7, 0.6e12},
};
// Row pitch (elements) of a stage's X and Y in shared memory: even, for 16-byte
// reads of two neighbours, and not a multiple of the 128-byte bank period, so
// that a run along k spreads over the banks.
constexpr int direct_ldx(int tr) { return (1 << tr) + 2; }
constexpr int direct_ldy(int tc) { return tc > 0 ? (1 << tc) + 2 : 1; }
constexpr int kNumDirectConfigs = (int)(sizeof(kDirectConfigs) / sizeof(kDirectConfigs[0]));

// Shape-dependent part of a direct step, fixed when it is planned.  X has the
// rows; legs are given by their bit positions in the operand.
struct DirectPlan {
  int config = 0;
  bool swap = false;       // X is the step's b operand (its small one), not a
  bool fold = false;       // the columns run over (pattern, column): X is shared by all patterns
  int cluster = 1;         // CTAs that split K
  int nr = 0, nk = 0, nc = 0;
  int64_t cols = 0;        // 2^nc, or PC * 2^nc with folded patterns
  int64_t col_tiles = 0;
  int n_rrest = 0, n_crest = 0;
  uint8_t rrest[32] = {0};           // X positions of the row legs above the tile
  uint8_t crest[32] = {0};           // Y positions of the column legs above the tile
  uint8_t kxrest[32] = {0}, kyrest[32] = {0};   // positions of the k legs above a stage
  // the tile's legs in the order of their position in the operand: position,
  // and which leg it is (0..31: row or column bit; 32 + q: k bit q)
  uint8_t xpos[16] = {0}, xleg[16] = {0};
  uint8_t ypos[16] = {0}, yleg[16] = {0};
  double seconds = 1e300;  // modelled time
};

// `xr`, `xk`: positions in X of the row and k legs (bit j of the row index is
// the leg at xr[j]); `yk`, `yc`: positions in Y of the k and column legs (at
// most 31 of each).  x_elems, y_elems: elements that the whole step reads of
// each operand.
struct DirectShape {
  int nr = 0, nk = 0, nc = 0;
  const int *xr = nullptr, *xk = nullptr, *yk = nullptr, *yc = nullptr;
  int64_t PC = 1;
  bool x_shared = false;   // every pattern reads X's pattern 0
  double x_elems = 0, y_elems = 0;
  bool bf16 = false;       // BF16x3 products: three multiply-adds for one
};
DirectPlan plan_direct(const DirectShape& s, bool fold);

// Parameters of one launch.
struct DirectParamsBase {
  int64_t x_pstride, y_pstride, c_pstride;
  int64_t cols, PC;
  uint32_t col_tiles;
  int nr, nk, nc, n_rrest, n_crest, fold, cluster;
  int mapX_mode, mapY_mode;      // 0 identity, 1 zero, 2 table
  int bf16;                      // 1: BF16x3 products
  int vec;                       // C and its pattern stride allow 16-byte stores of two rows
  uint8_t rrest[32], crest[32], kxrest[32], kyrest[32];
  // per bit of a stage's element index: what it adds to the source offset and
  // to the shared-memory slot (0 past the tile's legs)
  uint32_t xoff[16], xslot[16], yoff[16], yslot[16];
};
void direct_fill(const DirectPlan& d, int64_t PC, DirectParamsBase& q);

}  // namespace tn
