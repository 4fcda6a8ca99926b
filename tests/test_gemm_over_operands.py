"""tn_gemm_c64 with the result over one of its operands (C = A with N = K, C = B
with M = K, or one running into the other), in shapes that the direct kernel
takes when the buffers are apart and in ones it does not, on every engine.

Equal, bit for bit, to the same GEMM into a buffer of its own on the kernels
that read prepared copies (pair = 1; the CUDA-core engine has one kernel), and
close to NumPy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (M, N, K, patterns, element offset of C from A and from B; None: apart)
CASES = [
    (256, 128, 128, 1, 0, None),      # C = A, two row tiles of one A
    (128, 256, 128, 1, None, 0),      # C = B
    (64, 64, 64, 5, 0, None),
    (64, 64, 64, 5, None, 0),
    (4, 4, 4, 3, 0, None),
    (512, 64, 64, 3, 24, None),       # C starts inside A
    (64, 512, 64, 2, None, -24),      # C runs into B
    (2048, 512, 512, 1, 0, None),     # a tensor-core shape in either case
]


@pytest.mark.parametrize("engine", [1, 2, 3, 4], ids=["tf32x3", "simt", "bf16x3", "fp16x3"])
@pytest.mark.parametrize("case", CASES, ids=[f"M{c[0]}N{c[1]}K{c[2]}P{c[3]}a{c[4]}b{c[5]}" for c in CASES])
def test_result_over_an_operand(engine, case):
    import torch
    import paper_2111_03011_gb300 as tn
    M, N, K, P, over_a, over_b = case
    rng = np.random.default_rng(M + N + K + P)
    A, B = ((rng.normal(size=s) + 1j * rng.normal(size=s)).astype(np.complex64) for s in ((P, M, K), (P, K, N)))
    room = [torch.zeros(2 * P * max(M * K, K * N, M * N) + 64, dtype=torch.complex64, device="cuda") for _ in range(3)]

    def view(buf, start, shape):
        return buf[start:start + int(np.prod(shape))].view(shape)

    a, b = view(room[0], 32, A.shape), view(room[1], 32, B.shape)
    own = view(room[2], 32, (P, M, N))
    a.copy_(torch.from_numpy(A))
    b.copy_(torch.from_numpy(B))
    tn.tn_gemm_c64(a, b, own, engine=engine, pair=1)
    c = view(room[0], 32 + over_a, (P, M, N)) if over_a is not None else view(room[1], 32 + over_b, (P, M, N))
    tn.tn_gemm_c64(a, b, c, engine=engine)
    ref = A.astype(np.complex128) @ B.astype(np.complex128)
    assert torch.equal(torch.view_as_real(c), torch.view_as_real(own))
    assert np.linalg.norm(c.cpu().numpy() - ref) <= (1e-4 if engine == 3 else 1e-5) * np.linalg.norm(ref)
