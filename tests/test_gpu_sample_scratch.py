"""Draws whose prefix sums do not fit the scratch that can be had: the groups are
taken in windows, and the samples are the same, bit for bit."""
import numpy as np
import pytest

import circuit_inputs as ci

pytestmark = pytest.mark.gpu
NQ = 40


@pytest.fixture(scope="module")
def tn():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2111_03011_gb300 as m
    return m


def _head(tn, L, h):
    import torch
    rng = np.random.default_rng(L + h)
    H = (rng.normal(size=(L, 1 << h)) + 1j * rng.normal(size=(L, 1 << h))) * 2.0 ** (-(NQ + 1) / 2)
    H[::7] = 0.0
    oq = list(range(NQ - h, NQ))
    c = ci.make_grid_circuit(2, 2, 1, seed=1)
    c.n_qubits = NQ
    plan = tn.tn_plan(c, oq, ci.draw_tails(NQ, oq, L, seed=L + h), host_fold_log2=-1)
    buf = torch.zeros(H.shape, dtype=torch.complex128, device="cuda")
    head = tn.tn_head_create(plan, buf)
    buf.copy_(torch.from_numpy(H))
    tn.tn_head_set_fidelity(head, 1.0)
    torch.cuda.synchronize()
    return plan, head


# (groups, open qubits, samples): fewer and more samples than groups, a last
# round that ends inside, at and before a window
@pytest.mark.parametrize("method", [0, 2], ids=["exact", "frugal"])
@pytest.mark.parametrize("L,h,n", [(37, 8, 20), (37, 8, 37), (37, 8, 200), (64, 10, 1000), (5, 13, 7), (100, 6, 500),
                                   (1, 12, 50)])
def test_windows_of_groups_give_the_same_samples(tn, monkeypatch, method, L, h, n):
    plan, head = _head(tn, L, h)
    one = 8 * ((((1 << h) + 31) >> 5) + 1)                  # bytes of one group's prefix sums
    for f in (0.0, 0.4):
        want = tn.tn_sample_ex(head, n, f, 77, method=method)
        for groups in (1, 3, 8, 36):
            monkeypatch.setenv("TN_FAULT_INJECT", f"scratch:{groups * one + 7}")
            got = tn.tn_sample_ex(head, n, f, 77, method=method)
            monkeypatch.delenv("TN_FAULT_INJECT")
            assert np.array_equal(got, want)
    monkeypatch.setenv("TN_FAULT_INJECT", f"scratch:{one - 8}")
    with pytest.raises(tn.TNError) as e:                    # not even one group
        tn.tn_sample_ex(head, n, 0.0, 77, method=method)
    assert e.value.code == tn.TN_ERR_OOM


def test_server_takes_windows(tn, monkeypatch):
    cfg = ci.config_small(4, 4, 8, seed=3, n_open=8, L=48, n_cut_gates=0)
    plan = tn.tn_plan(cfg["circuit"], cfg["open_qubits"], cfg["tails"], cfg["edges"])
    head = tn.tn_head_create(plan)
    tn.tn_contract_slices(plan, 0, 1, head)
    want = [tn.tn_sample_ex(head, n, 0.0, 5, method=m) for n, m in ((30, 0), (500, 0), (500, 2))]
    sv = tn.tn_server_create(n_slots=2, hbm_budget_bytes=1 << 30)
    cid = tn.tn_server_add_circuit(sv, plan, 0, 1)
    monkeypatch.setenv("TN_FAULT_INJECT", f"scratch:{8 * 9 * 5}")
    tickets = [tn.tn_server_submit(sv, cid, tn.TN_REQ_SAMPLE, n, seed=5, method=m) for n, m in ((30, 0), (500, 0), (500, 2))]
    got = [tn.tn_server_wait(sv, t)[0] for t in tickets]
    monkeypatch.delenv("TN_FAULT_INJECT")
    tn.tn_server_free(sv)
    assert all(np.array_equal(a, b) for a, b in zip(got, want))
