"""Scratch that the library keeps between calls."""
import threading

import pytest

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
