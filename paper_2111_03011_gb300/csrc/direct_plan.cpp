// Host side of the direct contraction step (direct.cu): tile, tables and
// modelled time of a shape.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>
#include <vector>

#include "direct.h"

namespace tn {

namespace {

constexpr double kBytesPerSecond = 5.0e12;   // streaming reads and writes of the direct kernel
constexpr double kLaunchSeconds = 3.5e-6;    // a launch and its latency
constexpr int kSmCount = 152;
constexpr int kResident = 3;                 // CTAs of 256 threads per SM (registers and shared memory)
constexpr double kBusy = 2.0;                // CTAs per SM from which it runs near its full rate

// Legs of a tile sorted by position: (position, leg code).
void sorted_legs(const int* free_pos, int nfree, const int* k_pos, int nk, uint8_t* pos, uint8_t* leg) {
  std::vector<std::pair<int, int>> v;
  for (int j = 0; j < nfree; ++j) v.push_back({free_pos[j], j});
  for (int q = 0; q < nk; ++q) v.push_back({k_pos[q], 32 + q});
  std::sort(v.begin(), v.end());
  for (size_t i = 0; i < v.size(); ++i) {
    pos[i] = (uint8_t)v[i].first;
    leg[i] = (uint8_t)v[i].second;
  }
}

}  // namespace

// Tile choice: 64 rows, or 16 where the step has no more; 64, 32, 16, 4 or 1
// columns, the narrowest that covers them (a wider tile reads X fewer times
// and each value feeds more multiply-adds, but padding costs as much as work).
// 16-row tiles stop at 16 columns.
DirectPlan plan_direct(const DirectShape& s, bool fold) {
  DirectPlan d;
  if (s.nr > 31 || s.nc > 31 || s.nk > 31 || (fold && !s.x_shared)) return d;
  d.fold = fold;
  d.nr = s.nr;
  d.nk = s.nk;
  d.nc = s.nc;
  d.cols = fold ? s.PC << s.nc : 1LL << s.nc;
  const int tr = s.nr > 4 ? 6 : 4;
  const int tc = d.cols > 32 && tr == 6 ? 6 : d.cols > 16 && tr == 6 ? 5 : d.cols > 4 ? 4 : d.cols > 1 ? 2 : 0;
  for (int c = 0; c < kNumDirectConfigs; ++c)
    if (kDirectConfigs[c].tr == tr && kDirectConfigs[c].tc == tc) d.config = c;
  const DirectConfig& g = kDirectConfigs[d.config];
  const int trb = std::min(s.nr, g.tr), tkb = std::min(s.nk, g.tk), tcb = std::min(s.nc, g.tc);
  d.col_tiles = (d.cols + (1LL << g.tc) - 1) >> g.tc;
  sorted_legs(s.xr, trb, s.xk, tkb, d.xpos, d.xleg);
  sorted_legs(s.yc, tcb, s.yk, tkb, d.ypos, d.yleg);
  for (int j = trb; j < s.nr; ++j) d.rrest[d.n_rrest++] = (uint8_t)s.xr[j];
  for (int j = tcb; j < s.nc; ++j) d.crest[d.n_crest++] = (uint8_t)s.yc[j];
  for (int q = tkb; q < s.nk; ++q) {
    d.kxrest[q - tkb] = (uint8_t)s.xk[q];
    d.kyrest[q - tkb] = (uint8_t)s.yk[q];
  }
  // K over a cluster of CTAs while the launch leaves room on the chip and
  // every CTA keeps at least four stages
  const double tiles = (double)(d.col_tiles << d.n_rrest) * (fold ? 1.0 : (double)s.PC);
  const int64_t stages = 1LL << (s.nk - tkb);
  while (d.cluster < 8 && tiles * d.cluster * 2 <= kSmCount * kResident && stages >= 8 * d.cluster) d.cluster *= 2;
  const double ctas = tiles * d.cluster;
  if (ctas > 2147483647.0) return d;   // one grid dimension; left to the other forms
  const double padded = tiles * std::ldexp(1.0, g.tr + g.tc + s.nk);
  // fewer CTAs than the chip holds run at their share of the rate; X passes
  // through L2 once per column tile
  const double fill = std::min(1.0, ctas / (kSmCount * kBusy));
  const double c_elems = (double)s.PC * std::ldexp(1.0, s.nr + s.nc);
  const double l2 = 8.0 * s.x_elems * (double)(d.col_tiles - 1) / (2.0 * kBytesPerSecond);
  d.seconds = kLaunchSeconds + std::max(padded * (s.bf16 ? 3.5 : 1.0) / (g.rate * fill),
                                        8.0 * (s.x_elems + s.y_elems + c_elems) / (kBytesPerSecond * fill) + l2);
  return d;
}

// The shape-dependent launch parameters of a direct step.
void direct_fill(const DirectPlan& d, int64_t PC, DirectParamsBase& q) {
  q.cols = d.cols;
  q.col_tiles = (uint32_t)d.col_tiles;
  q.PC = PC;
  q.nr = d.nr;
  q.nk = d.nk;
  q.nc = d.nc;
  q.n_rrest = d.n_rrest;
  q.n_crest = d.n_crest;
  q.fold = d.fold;
  q.cluster = d.cluster;
  std::memcpy(q.rrest, d.rrest, sizeof(q.rrest));
  std::memcpy(q.crest, d.crest, sizeof(q.crest));
  std::memcpy(q.kxrest, d.kxrest, sizeof(q.kxrest));
  std::memcpy(q.kyrest, d.kyrest, sizeof(q.kyrest));
  const DirectConfig& g = kDirectConfigs[d.config];
  const int trb = std::min(d.nr, g.tr), tkb = std::min(d.nk, g.tk), tcb = std::min(d.nc, g.tc);
  const uint32_t ldx = direct_ldx(g.tr), ldy = direct_ldy(g.tc);
  for (int b = 0; b < 16; ++b) {
    q.xoff[b] = b < trb + tkb ? 1u << d.xpos[b] : 0u;
    q.xslot[b] = b < trb + tkb ? (d.xleg[b] < 32 ? 1u << d.xleg[b] : ldx << (d.xleg[b] - 32)) : 0u;
    q.yoff[b] = b < tcb + tkb ? 1u << d.ypos[b] : 0u;
    // the bits above the tile's legs count patterns side by side (folded)
    q.yslot[b] = b < tcb + tkb ? (d.yleg[b] < 32 ? 1u << d.yleg[b] : ldy << (d.yleg[b] - 32))
                 : b < g.tc + tkb ? 1u << (b - tkb) : 0u;
  }
}

}  // namespace tn
