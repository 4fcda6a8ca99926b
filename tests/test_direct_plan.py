"""Direct contraction steps on the host (no GPU): the bit scatters a launch is
given describe exactly the contraction of its operands' legs, whatever their
order, and stay inside the operands.

k_direct reads X at row, k and Y at k, column through the positions listed in
the step's "dp": the tile's legs in address order (xpos / xleg, ypos / yleg;
leg code 0..31 = row or column bit, 32 + q = k bit q) and the legs above the
tile (rrest, crest, kxrest, kyrest).  They are checked against the legs of the
three tensors, which the kernel never sees."""
import pytest

import circuit_inputs as ci


@pytest.fixture(scope="module")
def tn():
    import paper_2111_03011_gb300 as m
    return m


def _positions(pos, leg, free_rest, k_rest, tile_free, tile_k):
    """{row or column bit: position}, {k bit: position} of one operand."""
    assert list(pos) == sorted(pos) and len(pos) == len(leg)
    free = {c: x for x, c in zip(pos, leg) if c < 32}
    k = {c - 32: x for x, c in zip(pos, leg) if c >= 32}
    assert sorted(free) == list(range(min(tile_free, len(free)))) and sorted(k) == list(range(len(k)))
    assert (len(free) == tile_free or not free_rest) and (len(k) == tile_k or not k_rest)
    free.update({len(free) + i: x for i, x in enumerate(free_rest)})
    k.update({len(k) + i: x for i, x in enumerate(k_rest)})
    return free, k


def _check_direct(d, s):
    q = s["dp"]
    tr, tc, tk = q["tile"]
    vts = d["vts"]
    # the step's a operand is the larger of the pair that the order names
    big, sml = s["vt_a"], s["vt_b"]
    if vts[big]["P"] << len(vts[big]["legs"]) < vts[sml]["P"] << len(vts[sml]["legs"]):
        big, sml = sml, big
    x, y = (sml, big) if q["swap"] else (big, sml)
    lx, ly, lc = vts[x]["legs"], vts[y]["legs"], vts[s["vt_c"]]["legs"]
    rows, kx = _positions(q["xpos"], q["xleg"], q["rrest"], q["kxrest"], tr, tk)
    cols, ky = _positions(q["ypos"], q["yleg"], q["crest"], q["kyrest"], tc, tk)
    assert (len(rows), len(cols), len(kx), len(ky)) == (q["nr"], q["nc"], q["nk"], q["nk"])
    assert q["nr"] + q["nk"] == len(lx) and q["nc"] + q["nk"] == len(ly)
    # every leg of an operand is a row/column leg or a k leg, once
    assert sorted(list(rows.values()) + list(kx.values())) == list(range(len(lx)))
    assert sorted(list(cols.values()) + list(ky.values())) == list(range(len(ly)))
    # C = rows low, then columns; the k legs pair up
    assert [lx[rows[j]] for j in range(q["nr"])] + [ly[cols[j]] for j in range(q["nc"])] == lc
    assert [lx[kx[j]] for j in range(q["nk"])] == [ly[ky[j]] for j in range(q["nk"])]
    # columns of a launch, their tiles, and what folding needs
    assert q["cols"] == ((s["PC"] if q["fold"] else 1) << q["nc"])
    assert q["col_tiles"] == (q["cols"] + (1 << tc) - 1) >> tc
    if q["fold"]:
        assert (s["mapB"] if q["swap"] else s["mapA"])[0] == 1
    assert q["cluster"] in (1, 2, 4, 8) and (q["cluster"] == 1 or 1 << len(q["kxrest"]) >= 4 * q["cluster"])


CASES = [dict(r=4, c=4, m=8, seed=11, n_open=6, L=8, cut=2),
         dict(r=4, c=5, m=10, seed=13, n_open=8, L=24, cut=2), dict(r=4, c=6, m=10, seed=3, n_open=7, L=128, cut=0),
         dict(r=5, c=5, m=10, seed=4, n_open=3, L=1, cut=1)]


@pytest.mark.parametrize("gemm", [1, 3, 4])
@pytest.mark.parametrize("case", CASES, ids=[f"{c['r']}x{c['c']}m{c['m']}L{c['L']}" for c in CASES])
def test_direct_steps_describe_their_contraction(tn, case, gemm):
    cfg = ci.config_small(case["r"], case["c"], case["m"], seed=case["seed"], n_open=case["n_open"], L=case["L"],
                          n_cut_gates=case["cut"])
    seen = 0
    for fold in (-1, 0):
        p = tn.tn_plan(cfg["circuit"], cfg["open_qubits"], cfg["tails"], cfg["edges"], host_only=True, gemm=gemm,
                       host_fold_log2=fold)
        d = tn.tn_plan_describe(p)
        for s in d["steps"]:
            if s["direct"]:
                assert s["kind"] == 0
                _check_direct(d, s)
                seen += 1
    assert seen > 0
    # plans that ask for the GEMM form, and the plain CUDA-core engine, have none
    for kw in (dict(gemm=gemm, small_max_bits=-1), dict(gemm=gemm, small_max_bits=2), dict(gemm=2)):
        p = tn.tn_plan(cfg["circuit"], cfg["open_qubits"], cfg["tails"], cfg["edges"], host_only=True, **kw)
        assert not any(s["direct"] for s in tn.tn_plan_describe(p)["steps"])
