"""A tn_contract_batch that fails on the way leaves every head as it was, on the
path of a first submission (launched directly: empty heads of the library's own)
and on the captured one (heads that hold something, or that the caller can
write), and the same batch is accepted afterwards."""
import numpy as np
import pytest

import circuit_inputs as ci

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2111_03011_gb300 as tn
    cfgs = [ci.config_small(4, 4, 6 + i, seed=50 + i, n_open=5, L=6, n_cut_gates=i % 2, tail_seed=60 + i) for i in range(4)]
    plans = [tn.tn_plan(c["circuit"], c["open_qubits"], c["tails"], c["edges"], gemm=[1, 4][i % 2])
             for i, c in enumerate(cfgs)]
    ends = [1 << tn.tn_plan_get_stats(p)["n_sliced"] for p in plans]
    bits = [np.array([int(t) | (mu << 11) for t in c["tails"] for mu in range(32)], dtype=np.uint64) for c in cfgs]
    assert ends == [1, 4, 1, 4]
    return tn, plans, ends, bits


def _plain(tn, plan, bits, *ranges):
    h = tn.tn_head_create(plan)
    for b, e in ranges:
        tn.tn_contract_slices(plan, b, e, h)
    return tn.tn_amplitudes(h, bits)


def _failing(tn, monkeypatch, fault, *args):
    monkeypatch.setenv("TN_FAULT_INJECT", fault)
    with pytest.raises(tn.TNError) as e:
        tn.tn_contract_batch(*args)
    monkeypatch.delenv("TN_FAULT_INJECT")
    assert "injected" in str(e.value)


@pytest.mark.parametrize("fault", ["slice:0", "slice:1", "slice:3"])
@pytest.mark.parametrize("own", [True, False], ids=["own", "caller's"])
def test_first_submission_fails(setup, monkeypatch, fault, own):
    import torch
    tn, plans, ends, bits = setup
    bufs = [torch.zeros((6, 32), dtype=torch.complex128, device="cuda") for _ in plans]
    heads = [tn.tn_head_create(p) if own else tn.tn_head_create(p, b) for p, b in zip(plans, bufs)]
    batch = (plans, [(0, e) for e in ends], heads)
    _failing(tn, monkeypatch, fault, *batch)        # items before the failing slice were launched
    for h, b in zip(heads, bits):
        assert tn.tn_head_fidelity(h)[1] == 0
        assert not tn.tn_amplitudes(h, b).any()
    for _ in range(2):                              # accepted again, then replayed
        tn.tn_contract_batch(*batch)
        for p, e, h, b in zip(plans, ends, heads, bits):
            assert np.array_equal(tn.tn_amplitudes(h, b), _plain(tn, p, b, (0, e)))
            tn.tn_head_reset(h)


def test_failure_leaves_what_heads_hold(setup, monkeypatch):
    tn, plans, ends, bits = setup
    heads = [tn.tn_head_create(p) for p in plans]
    for i in (1, 3):
        tn.tn_contract_slices(plans[i], 0, 1, heads[i])
    batch = (plans, [(0, 1), (1, 4), (0, 1), (1, 4)], heads)
    before = [tn.tn_amplitudes(h, b) for h, b in zip(heads, bits)]
    _failing(tn, monkeypatch, "slice:2", *batch)
    for i, (h, b) in enumerate(zip(heads, bits)):
        assert np.array_equal(tn.tn_amplitudes(h, b), before[i]) and tn.tn_head_fidelity(h)[1] == i % 2
    tn.tn_contract_batch(*batch)
    for i, (p, h, b) in enumerate(zip(plans, heads, bits)):
        want = _plain(tn, p, b, (0, 1), (1, 4)) if i % 2 else _plain(tn, p, b, (0, 1))
        assert np.array_equal(tn.tn_amplitudes(h, b), want)
