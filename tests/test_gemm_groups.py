"""Pattern groups of tensor-core GEMM steps with gathered A patterns, on the
host: every pattern is in exactly one group, a group's patterns read one A
pattern, and the runs that the tile order uses are those of equal A patterns.
The kernel's tile decoding is repeated here: every (m-tile, n-tile, group) once."""
import numpy as np
import pytest

import circuit_inputs as ci

ST_GEMM_TC = 3
NONE = 0xFFFFFFFF


@pytest.fixture(scope="module")
def tn():
    import paper_2111_03011_gb300 as m
    return m


def _decode(t, tilesM, tilesN, runs):
    """tile_coords of gemm_tc.cu with a group table."""
    gm = min(8, tilesM)
    mgroups = tilesM // gm
    u, r = divmod(t, gm * tilesN)
    first, count = runs[u // mgroups]
    w = u - first * mgroups
    mg, g = divmod(w, count)
    tn_, mi = divmod(r, gm)
    return first + g, mg * 8 + mi, tn_


@pytest.mark.parametrize("gemm", [1, 3, 4])
@pytest.mark.parametrize("L,m", [(24, 10), (100, 9), (256, 8)])
def test_groups_cover_the_patterns(tn, gemm, L, m):
    cfg = ci.config_small(4, 6, m, seed=13, n_open=6, L=L, n_cut_gates=1)
    seen = folded = 0
    for small in (-1, 0):
        p = tn.tn_plan(cfg["circuit"], cfg["open_qubits"], cfg["tails"], cfg["edges"], host_only=True, gemm=gemm,
                       small_max_bits=small, host_fold_log2=-1)
        d = tn.tn_plan_describe(p, with_data=True)
        meta = np.asarray(d["meta"], dtype=np.int64)
        for s in d["steps"]:
            fold, ng, off = s["grp"]
            if s["kind"] != ST_GEMM_TC or s["mapA"][0] != 2 or s["PA"] >= s["PC"]:
                assert fold == 0
                continue
            seen += 1
            folded += fold > 1
            n2 = 2 << s["nn"]
            assert fold == 1 or (n2 >= 16 and n2 * fold <= 256)
            assert off % 2 == 0 and off + (ng * fold + 1) // 2 * 2 + 2 * ng <= meta.size
            ids = meta[off:off + ng * fold].reshape(ng, fold)
            runs = meta[off + (ng * fold + 1) // 2 * 2:][:2 * ng].reshape(ng, 2)
            mapA = meta[s["mapA"][1]:s["mapA"][1] + s["PC"]]
            real = ids[ids != NONE]
            assert sorted(real) == list(range(s["PC"]))
            assert (ids[:, 0] != NONE).all()
            for g in range(ng):
                a = {int(mapA[x]) for x in ids[g] if x != NONE}
                assert len(a) == 1
                first, count = runs[g]
                assert first <= g < first + count <= ng
                assert all(mapA[ids[x, 0]] == mapA[ids[g, 0]] for x in range(first, first + count))
                assert first == 0 or mapA[ids[first - 1, 0]] != mapA[ids[g, 0]]
            for rows in (128, 256):
                tilesM = max(1, (1 << s["nm"]) // rows)
                tilesN = 1 if fold > 1 else max(1, n2 // 256)
                if tilesM * tilesN * ng > 20000:
                    continue
                tiles = {_decode(t, tilesM, tilesN, runs) for t in range(tilesM * tilesN * ng)}
                assert tiles == {(g, a, b) for g in range(ng) for a in range(tilesM) for b in range(tilesN)}
    assert seen > 0 and folded > 0
