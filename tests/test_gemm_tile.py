"""Which tile a tensor-core GEMM runs on.  The rule is checked on the CPU, from
its own source, over every kind of shape: a width that a kernel exists for, no
wider than the columns need, folds that the kernels accept, merges that keep the
work; and the modelled time is that of the merged, joined or grouped launch.
Merged rows are compared with NumPy on the GPU.  Plans with narrow gathered steps (a table of pattern groups, fewer than
16 real columns) are contracted on the GPU and compared with the state vector."""
import os
import subprocess

import numpy as np
import pytest

import circuit_inputs as ci
import oracle as O

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2111_03011_gb300", "csrc")

CHECK = r"""
#include "gemm_tile.h"
#include <algorithm>
#include <cstdio>
#include <initializer_list>
using namespace tn;
int main() {
  long bad = 0, seen = 0;
  for (int nm = 0; nm <= 12; ++nm) for (int nn = 0; nn <= 10; ++nn)
  for (int64_t PC : {1, 2, 3, 7, 64, 147}) for (int ma = 0; ma < 3; ++ma) for (int mb = 0; mb < 3; ++mb)
  for (int h16 = 0; h16 < 3; ++h16) for (int pair = -1; pair <= 0; ++pair) for (int cap : {32, 64, 128, 256})
  for (int fold = 0; fold <= 16; fold = fold ? fold * 2 : 1) {
    const int64_t N2 = 2LL << nn;
    if (fold && (ma != 2 || (fold > 1 && (N2 < 16 || N2 * fold > 256)))) continue;   // tables as the planner makes them
    GemmShape s;
    s.M = 1LL << nm; s.N = 1LL << nn; s.PC = PC;
    s.PA = ma == 0 ? PC : ma == 1 ? 1 : 2;
    s.PB = mb == 0 ? PC : mb == 1 ? 1 : 2;
    s.mapA_mode = ma; s.mapB_mode = mb; s.h16 = h16; s.pair = pair; s.tile_cap = cap;
    s.grp_fold = fold; s.n_groups = fold ? (PC + fold - 1) / fold : 0;
    const GemmForm f = gemm_form(s, kGemmSMs);
    ++seen;
    bool ok = f.bn == 16 || f.bn == 32 || f.bn == 64 || f.bn == 128 || f.bn == 256;
    ok = ok && f.bn <= std::max(cap, 16);
    // as narrow as the columns that a tile can have allow
    ok = ok && (f.bn == 16 || f.bn / 2 < 2 * f.N * f.fold);
    ok = ok && (f.fold == 1 || (f.bn == 2 * f.N * f.fold && 2 * f.N >= 16 && (f.mapA_mode == 1 || f.grouped)));
    ok = ok && f.grouped == (fold > 0 && cap == 256) && (!f.grouped || f.fold == fold);
    ok = ok && (!f.paired || (f.bn == 256 && f.M >= 256 && pair == 0 && f.fold % (f.fold > 1 ? 2 : 1) == 0));
    ok = ok && f.M * f.N * f.PC == s.M * s.N * s.PC;
    ok = ok && (f.sub_log2 < 0 || (2LL << nn) == 1LL << f.sub_log2);
    bad += !ok;
  }
  std::printf("%ld %d\n", bad, seen > 100000);
  return 0;
}
"""


def test_tile_rule(tmp_path):
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(CHECK)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), os.path.join(CSRC, "gemm_tile.cpp"), "-o",
                    str(exe)], check=True)
    assert subprocess.run([str(exe)], stdout=subprocess.PIPE, check=True).stdout == b"0 1\n"


MODEL = r"""
#include "gemm_tile.h"
#include <cstdio>
#include <initializer_list>
using namespace tn;
static double t(const GemmShape& s) {
  return tc_seconds(gemm_form(s, kGemmSMs), 9, 1e6, 1e5, 1e6, s.h16 != 0);
}
int main() {
  int bad = 0;
  for (int h16 = 0; h16 < 2; ++h16)
    for (int64_t P : {2, 64, 400, 3000}) for (int64_t M : {1, 2, 16}) for (int64_t N : {1, 4, 64, 512}) {
      GemmShape s, r;
      s.h16 = r.h16 = h16;
      // own A, shared B: one GEMM of P M rows
      s.M = M; s.N = N; s.PA = s.PC = P; s.mapA_mode = 0; s.mapB_mode = 1;
      r.M = P * M; r.N = N;
      bad += t(s) != t(r);
      // shared A, own narrow B: one GEMM of P N columns
      if (2 * N < 16) {
        s = GemmShape(); r = GemmShape();
        s.h16 = r.h16 = h16;
        s.M = 4096; s.N = N; s.PB = s.PC = P; s.mapB_mode = 0;
        r.M = 4096; r.N = P * N;
        bad += t(s) != t(r);
      }
      // gathered A in groups of 4: as many patterns of 4 N columns
      if (2 * N >= 16 && 8 * N <= 256) {
        s = GemmShape(); r = GemmShape();
        s.h16 = r.h16 = h16;
        s.M = 2048; s.N = N; s.PA = 7; s.PB = 9; s.PC = P; s.mapA_mode = s.mapB_mode = 2;
        s.grp_fold = 4; s.n_groups = (P + 3) / 4 + 3;
        r.M = 2048; r.N = 4 * N; r.PA = 7; r.PB = 9; r.PC = s.n_groups; r.mapA_mode = r.mapB_mode = 2;
        bad += t(s) != t(r);
      }
    }
  std::printf("%d\n", bad);
  return 0;
}
"""


def test_modelled_time_is_that_of_the_launch(tmp_path):
    src, exe = tmp_path / "model.cpp", tmp_path / "model"
    src.write_text(MODEL)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), os.path.join(CSRC, "gemm_tile.cpp"), "-o",
                    str(exe)], check=True)
    assert subprocess.run([str(exe)], stdout=subprocess.PIPE, check=True).stdout == b"0\n"


CIRCUITS = [dict(r=4, c=4, m=8, L=24, seed=0), dict(r=4, c=5, m=10, L=50, seed=1), dict(r=3, c=6, m=9, L=40, seed=2)]
IDS = [f"{c['r']}x{c['c']}" for c in CIRCUITS]


def _plan(case, gemm, **kw):
    import paper_2111_03011_gb300 as tn
    cfg = ci.config_small(case["r"], case["c"], case["m"], seed=case["seed"], n_open=6, L=case["L"], n_cut_gates=1)
    return tn, cfg, tn.tn_plan(cfg["circuit"], cfg["open_qubits"], cfg["tails"], cfg["edges"], gemm=gemm,
                               small_max_bits=-1, host_fold_log2=-1, **kw)


@pytest.mark.parametrize("gemm", [1, 3, 4])
@pytest.mark.parametrize("case", CIRCUITS, ids=IDS)
def test_narrow_gathered_steps_run_on_narrow_tiles(case, gemm):
    tn, _, p = _plan(case, gemm, host_only=True)
    d = tn.tn_plan_describe(p)
    assert [t[0] for t in d["gemm_tiles"]] == [i for i, s in enumerate(d["steps"]) if s["kind"] == 3]
    narrow = 0
    for i, _, n2, bn, fold, _, grouped in d["gemm_tiles"]:
        s = d["steps"][i]
        if grouped and 2 << s["nn"] < 16:
            assert (n2, bn, fold) == (2 << s["nn"], 16, 1)
            narrow += 1
    assert narrow > 0


@pytest.mark.gpu
@pytest.mark.parametrize("gemm", [1, 3, 4])
@pytest.mark.parametrize("case", CIRCUITS, ids=IDS)
def test_plans_with_narrow_gathered_steps(case, gemm):
    tn, cfg, p = _plan(case, gemm)
    oq, tails = cfg["open_qubits"], cfg["tails"]
    ref = O.sparse_state_from_vector(O.sliced_statevector(cfg["circuit"], [(g, l) for (g, l, k, v) in cfg["edges"]]),
                                     oq, tails)
    head = tn.tn_head_create(p)
    tn.tn_contract_slices(p, 0, 1 << tn.tn_plan_get_stats(p)["n_sliced"], head)
    bits = np.array([O.bitstring_index(int(t), oq, mu) for t in tails for mu in range(1 << len(oq))], np.uint64)
    H = tn.tn_amplitudes(head, bits).reshape(len(tails), -1)
    assert np.linalg.norm(H - ref) <= (1e-4 if gemm == 3 else 1e-5) * np.linalg.norm(ref)


# (M, N, K, patterns): ragged last row tiles of one CTA and of pairs, one row a
# pattern, columns narrower than 16 and K = 2
ROWS = [(64, 16, 32, 3), (128, 128, 64, 3), (1, 64, 64, 217), (2, 64, 1024, 130), (256, 256, 16, 5), (8, 2, 128, 77),
        (16, 512, 2, 50)]


@pytest.mark.gpu
@pytest.mark.parametrize("gemm", [1, 3, 4])
@pytest.mark.parametrize("pair", [1, -1])
@pytest.mark.parametrize("shape", ROWS, ids=str)
def test_merged_rows(gemm, pair, shape):
    """Every pattern its own A, one B for all.  Relative L2 as for any GEMM: 1e-5
    (3xTF32, FP16x3) or 1e-4 (BF16x3)."""
    import torch
    import paper_2111_03011_gb300 as tn
    M, N, K, P = shape
    rng = np.random.default_rng(M + N + K + P)
    A, B = ((rng.normal(size=s) + 1j * rng.normal(size=s)).astype(np.complex64) for s in ((P, M, K), (1, K, N)))
    ref = A.astype(np.complex128) @ B.astype(np.complex128)
    buf = torch.full((P * M * N + 2,), float("nan"), dtype=torch.complex64, device="cuda")
    c = buf[1:-1].view(P, M, N)
    tn.tn_gemm_c64(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), c, engine=gemm, pair=pair)
    assert np.linalg.norm(c.cpu().numpy() - ref) <= (1e-4 if gemm == 3 else 1e-5) * np.linalg.norm(ref)
    rest = buf.cpu().numpy()
    assert np.isnan(rest[0]) and np.isnan(rest[-1])
