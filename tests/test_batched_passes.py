"""Steps launched once for a chunk of passes: which ones, and where their
copies lie (CPU); chunks give the same bits as passes one by one (GPU)."""
import numpy as np
import pytest

import circuit_inputs as ci


@pytest.fixture(scope="module")
def tn():
    import paper_2111_03011_gb300 as m
    return m


def _cfgs():
    base = ci.config_small(4, 4, 8, seed=11, n_open=6, L=8, n_cut_gates=2)
    yield "4x4", base, {}
    yield "4x4 unfolded", base, dict(host_fold_log2=-1)
    yield "folded whole", base, dict(host_fold_log2=16)
    yield "4x5", ci.config_small(4, 5, 10, seed=13, n_open=7, L=24, n_cut_gates=2), dict(host_fold_log2=6)
    yield "auto-sliced", ci.config_small(4, 5, 10, seed=13, n_open=6, L=24, n_cut_gates=1), dict(
        max_log2_elements=14, auto_slice=12)


CFGS = list(_cfgs())
IDS = [c[0] for c in CFGS]


@pytest.mark.parametrize("cfg", CFGS, ids=IDS)
@pytest.mark.parametrize("gemm", [1, 3, 4])
def test_batched_steps_and_their_copies(tn, cfg, gemm):
    _, c, kw = cfg
    p = tn.tn_plan(c["circuit"], c["open_qubits"], c["tails"], c["edges"], host_only=True, gemm=gemm, **kw)
    d = tn.tn_plan_describe(p, with_data=True)
    most, stride = d["batch"]
    assert 1 <= most <= 64 and most <= 1 << (d["n_sliced"] + d["n_internal"])
    base = d["workspace_bytes"] - most * stride
    steps, bufs = d["steps"], d["bufs"]
    written = {s["c"][1] for s in steps if s["batch"]}
    for s in steps:
        if s["batch"]:
            assert s["kind"] == 0 and s["PC"] << s["rC"] <= 1 << 18
            for kind, rid in (s["a"], s["b"]):
                assert rid in written if kind == 1 else len(d["leaves"][rid]["var_slice_bits"]) <= 8
    for i, (off, nbytes, first, last) in enumerate(bufs):
        if i in written:
            assert base <= off and off + nbytes <= base + stride
        else:
            assert off + nbytes <= base
    # what a pass's own steps (or the accumulation) read stays until the chunk ends
    readers = [r for s in steps if not s["batch"] for r in (s["a"], s["b"])] + [d["final"]["ref"]]
    for kind, rid in readers:
        if kind == 1 and rid in written:
            assert bufs[rid][3] == len(steps)


def _head(tn, plan, calls, graph=False):
    import torch
    st = tn.tn_plan_get_stats(plan)
    buf = torch.zeros((st["n_tails"], 1 << st["n_open"]), dtype=torch.complex128, device="cuda")
    head = tn.tn_head_create(plan, buf)
    for b, e in calls:
        (tn.tn_contract_slices_graph if graph else tn.tn_contract_slices)(plan, b, e, head)
    torch.cuda.synchronize()
    return buf.cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("cfg", CFGS, ids=IDS)
@pytest.mark.parametrize("gemm", [1, 2, 3, 4])
def test_chunks_equal_single_passes(tn, cfg, gemm):
    _, c, kw = cfg
    p = tn.tn_plan(c["circuit"], c["open_qubits"], c["tails"], c["edges"], gemm=gemm, **kw)
    n = 1 << tn.tn_plan_get_stats(p)["n_sliced"]
    one = _head(tn, p, [(s, s + 1) for s in range(n)])
    assert np.abs(one).max() > 0
    assert np.array_equal(one, _head(tn, p, [(0, n)]))
    assert np.array_equal(one, _head(tn, p, [(0, n)], graph=True))
    part = _head(tn, p, [(s, s + 1) for s in range(1, n)])
    assert np.array_equal(part, _head(tn, p, [(1, n)])) and not np.array_equal(part, one)
    prof = tn.tn_head_create(p)
    tn.tn_profile_slices(p, 0, n, prof)          # launches every step of every pass
    assert tn.tn_head_norm(prof) == pytest.approx(np.sum(np.abs(one) ** 2), rel=1e-12)


@pytest.mark.gpu
def test_failure_inside_a_chunk_keeps_the_passes_before_it(tn, monkeypatch):
    c = CFGS[0][1]
    p = tn.tn_plan(c["circuit"], c["open_qubits"], c["tails"], c["edges"])
    import torch
    st = tn.tn_plan_get_stats(p)
    buf = torch.zeros((st["n_tails"], 1 << st["n_open"]), dtype=torch.complex128, device="cuda")
    head = tn.tn_head_create(p, buf)
    monkeypatch.setenv("TN_FAULT_INJECT", "slice:5")
    with pytest.raises(tn.TNError):
        tn.tn_contract_slices(p, 0, 16, head)
    monkeypatch.delenv("TN_FAULT_INJECT")
    assert tn.tn_head_fidelity(head)[1] == 5
    tn.tn_contract_slices(p, 5, 16, head)
    torch.cuda.synchronize()
    assert np.array_equal(buf.cpu().numpy(), _head(tn, p, [(0, 16)]))


@pytest.mark.gpu
def test_batches_first_seen_and_replayed(tn, monkeypatch):
    """A batch's first submission (branch streams), its second (captured) and
    later ones (replayed, also after enough other batches to drop its graph)
    give the heads of plain calls, bit for bit; a failing submission leaves every
    head as it was."""
    import torch
    cfgs = [ci.config_small(4, 4, 6 + i, seed=20 + i, n_open=5, L=6, n_cut_gates=i % 2, tail_seed=30 + i)
            for i in range(12)]
    plans = [tn.tn_plan(c["circuit"], c["open_qubits"], c["tails"], c["edges"], gemm=[1, 4][i % 2])
             for i, c in enumerate(cfgs)]
    ends = [1 << tn.tn_plan_get_stats(p)["n_sliced"] for p in plans]
    ref = [_head(tn, p, [(0, e)]) for p, e in zip(plans, ends)]
    bufs = [torch.zeros(r.shape, dtype=torch.complex128, device="cuda") for r in ref]
    heads = [tn.tn_head_create(p, b) for p, b in zip(plans, bufs)]

    def submit(idx):
        for i in idx:
            tn.tn_head_reset(heads[i])
        tn.tn_contract_batch([plans[i] for i in idx], [(0, ends[i]) for i in idx], [heads[i] for i in idx])
        torch.cuda.synchronize()
        for i in idx:
            assert np.array_equal(bufs[i].cpu().numpy(), ref[i])

    batches = [[i, (i + 1) % 12, (i + 5) % 12] for i in range(10)]
    for _ in range(3):
        for b in batches:
            submit(b)
    submit(list(range(12)))
    for i in range(3):
        tn.tn_head_reset(heads[i])
    torch.cuda.synchronize()
    monkeypatch.setenv("TN_FAULT_INJECT", "slice:0")
    with pytest.raises(tn.TNError):
        tn.tn_contract_batch(plans[:3], [(0, e) for e in ends[:3]], heads[:3])
    monkeypatch.delenv("TN_FAULT_INJECT")
    torch.cuda.synchronize()
    assert all(float(b.abs().max()) == 0.0 for b in bufs[:3])
    assert all(tn.tn_head_fidelity(h)[1] == 0 for h in heads[:3])
    submit([0, 1, 2])


@pytest.mark.parametrize("gemm", [1, 3, 4])
def test_joint_preparations_share_no_memory(tn, gemm):
    """A GEMM's permute and the B preparation right after it may run in one launch:
    B's result and everything the permute reads or writes are apart."""
    seen = 0
    for c, kw in ((ci.config_small(4, 6, 10, seed=13, n_open=6, L=24, n_cut_gates=1), {}),
                  (ci.config_small(4, 5, 10, seed=13, n_open=7, L=24, n_cut_gates=1), dict(small_max_bits=-1)),
                  (ci.config_sliced30(), dict(order_trials=64, max_log2_elements=31))):
        p = tn.tn_plan(c["circuit"], c["open_qubits"], c["tails"], c["edges"], host_only=True, gemm=gemm, **kw)
        d = tn.tn_plan_describe(p)
        for x, y in zip(d["steps"], d["steps"][1:]):
            if x["kind"] != 1 or y["kind"] != 2 or x["contraction"] != y["contraction"]:
                continue
            seen += 1
            assert y["a"] != x["c"]
            o, n = d["bufs"][y["c"][1]][:2]
            for kind, rid in (x["a"], x["c"], y["a"]):
                if kind == 1:
                    o2, n2 = d["bufs"][rid][:2]
                    assert o + n <= o2 or o2 + n2 <= o
    assert seen > 5
