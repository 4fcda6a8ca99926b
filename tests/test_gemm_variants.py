"""The tile variants that a GEMM step offers to a tuner are the forms that it
launches: no two alike, and one-CTA tiles wherever the step runs on CTA pairs
(3xTF32, merged rows, joined columns and grouped patterns among them)."""
import pytest

import circuit_inputs as ci


def _plans(tn, gemm):
    yield ci.config_small(5, 5, 12, seed=4, n_open=6, L=99, n_cut_gates=1), {}
    yield ci.config_small(4, 6, 10, seed=3, n_open=7, L=200, n_cut_gates=0), dict(small_max_bits=-1)
    yield ci.config_small(4, 6, 8, seed=1, n_open=6, L=256, n_cut_gates=1), dict(small_max_bits=-1, host_fold_log2=-1)


@pytest.mark.parametrize("gemm", [1, 3, 4])
def test_variants_are_the_launched_forms(gemm):
    import paper_2111_03011_gb300 as tn
    n_paired = n_grouped = 0
    for cfg, kw in _plans(tn, gemm):
        p = tn.tn_plan(cfg["circuit"], cfg["open_qubits"], cfg["tails"], cfg["edges"], host_only=True, gemm=gemm, **kw)
        default = tn.tn_plan_describe(p)["gemm_tiles"]
        counts = {t[0]: tn.tn_plan_step_variants(p, t[0])[0] for t in default}
        forms = {i: [] for i in counts}
        for v in range(max(counts.values())):
            for i, n in counts.items():
                if v < n:
                    tn.tn_plan_set_step_variant(p, i, v)
            for t in tn.tn_plan_describe(p)["gemm_tiles"]:
                if v < counts[t[0]]:
                    forms[t[0]].append(tuple(t))
        for t in default:
            f = forms[t[0]]
            assert f[0] == tuple(t) and len(set(f)) == len(f)
            paired, grouped = t[5], t[6]
            n_grouped += grouped and paired
            if paired:
                n_paired += 1
                assert any(x[3] == 256 and not x[5] and x[6] == grouped for x in f)
    assert n_paired > 0 and n_grouped > 0
