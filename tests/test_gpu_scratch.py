"""Scratch that the library keeps between calls: it stands in no other call's way."""
import threading

import numpy as np
import pytest

import circuit_inputs as ci

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tn():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2111_03011_gb300 as m
    return m


def _operands(M, N, K):
    import torch
    return [torch.ones(s, dtype=torch.complex64, device="cuda") for s in ((1, M, K), (1, K, N), (1, M, N))]


def test_scratch_beyond_the_pool_leaves_a_capture_alone(tn):
    """The planes of 2^14 x 2^13 in 3xTF32 are above what the pool keeps (2 GiB):
    allocated and freed within the call, beside a thread-local capture of another
    thread (in global mode CUDA allows no thread to synchronise a stream)."""
    import torch
    a, b, c = _operands(1 << 14, 16, 1 << 13)
    x = torch.zeros(8, device="cuda")
    other = torch.cuda.Stream()
    failed = []

    def call():
        try:
            tn.tn_gemm_c64(a, b, c, engine=1, pair=1, stream=other)
        except Exception as e:
            failed.append(e)

    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        x.add_(1)
        t = threading.Thread(target=call)
        t.start()
        t.join()
        x.add_(2)
    assert not failed
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [6.0] * 8
    assert float((c - (1 << 13)).abs().max()) <= 1e-5 * (1 << 13)


def test_server_counts_kept_scratch_as_free(tn):
    """700 MiB free beside 1 GiB of kept scratch: a request whose head needs the
    server's reserve of 1 GiB is admitted (the scratch is given back), and nothing
    else had to go."""
    import torch
    cfg = ci.config_small(4, 4, 8, seed=11, n_open=6, L=8, n_cut_gates=1)
    plan = tn.tn_plan(cfg["circuit"], cfg["open_qubits"], cfg["tails"], cfg["edges"])
    n = 1 << tn.tn_plan_get_stats(plan)["n_sliced"]
    head = tn.tn_head_create(plan)
    tn.tn_contract_slices(plan, 0, n, head)
    bits = np.array([int(t) | (mu << 10) for t in cfg["tails"] for mu in range(64)], dtype=np.uint64)
    want = tn.tn_amplitudes(head, bits)
    sv = tn.tn_server_create(n_slots=2, hbm_budget_bytes=1 << 30)
    cid = tn.tn_server_add_circuit(sv, plan, 0, n)
    tn.tn_gemm_c64(*_operands(1 << 13, 16, 1 << 13), engine=1, pair=1)     # planes of 1 GiB
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (700 << 20), dtype=torch.uint8, device="cuda")
    got = []
    ticket = tn.tn_server_submit(sv, cid, tn.TN_REQ_AMPLITUDES, 0, bitstrings=bits)
    t = threading.Thread(target=lambda: got.append(tn.tn_server_wait(sv, ticket)[0]))
    t.start()
    t.join(20)
    waited = t.is_alive()
    del fill
    torch.cuda.empty_cache()                   # a request that waits for memory has it now
    t.join(60)
    st = tn.tn_server_get_stats(sv)
    tn.tn_server_free(sv)
    assert np.array_equal(got[0], want) and not waited and st["evictions"] == 0
