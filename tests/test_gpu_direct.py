"""The direct contraction kernel on the GPU, through tn_gemm_c64 with shapes
that it takes (small or narrow), against NumPy complex128.

Edges of every tile: fewer rows or columns than the tile, one column, ragged
last column tiles of folded patterns, K below a stage and K long enough to be
split over a cluster, gather tables, and an output that starts on 8 but not on
16 bytes.

Tolerance: each output is a sum of K products accumulated in FP32, so its
rounding errors are at most about 2 sqrt(K) + 4 units of 2^-24 of the root of
the summed squares (independent errors; 4 roundings per complex product)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (M, N, K, PA, PB, PC, mapA, mapB): rows are N, columns M (or patterns x M)
SHAPES = [
    (1, 1, 2, 1, 1, 1, None, None),             # one output
    (64, 1, 4, 1, 1, 1, None, None),            # one row
    (1, 64, 16, 1, 1, 1, None, None),           # one column: (64, 1) tile
    (1, 8, 64, 1, 1, 1, None, None),            # (16, 1) tile
    (4, 16, 512, 1, 1, 1, None, None),          # (16, 4) tile, K split over a cluster
    (16, 16, 8192, 1, 1, 1, None, None),        # (16, 16) tile, cluster of 8
    (4, 128, 256, 3, 3, 3, None, None),         # (64, 4) tile
    (16, 256, 64, 2, 2, 2, None, None),         # (64, 16) tile
    (32, 64, 128, 1, 5, 5, None, None),         # (64, 32) tile
    (256, 128, 32, 1, 1, 1, None, None),        # (64, 64) tiles
    (2, 64, 256, 53, 1, 53, None, None),        # folded: 106 columns, ragged last tile
    (128, 64, 8, 7, 1, 7, None, None),          # folded: two tiles per pattern
    (8, 32, 16, 1, 1, 11, [0] * 11, [0] * 11),  # gather tables to one pattern
    (64, 64, 16, 5, 4, 9, [4, 0, 1, 1, 2, 3, 0, 4, 2], [3, 3, 0, 1, 2, 0, 1, 2, 3]),
    (512, 64, 8, 16, 8, 51, [i % 16 for i in range(51)], [i % 8 for i in range(51)]),
]


@pytest.fixture(scope="module")
def tn():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2111_03011_gb300 as m
    return m


@pytest.mark.parametrize("shift", [0, 1], ids=["aligned", "8-byte"])
@pytest.mark.parametrize("shape", SHAPES, ids=[f"M{s[0]}N{s[1]}K{s[2]}P{s[3]}x{s[4]}x{s[5]}" for s in SHAPES])
@pytest.mark.parametrize("engine", [1, 4], ids=["tf32x3", "fp16x3"])
def test_direct_kernel_against_numpy(tn, engine, shape, shift):
    import torch
    M, N, K, PA, PB, PC, ma, mb = shape
    rng = np.random.default_rng(M * 7 + N * 3 + K + PA + 5 * PB + PC)
    A, B = (rng.normal(size=s) + 1j * rng.normal(size=s) for s in ((PA, M, K), (PB, K, N)))
    A, B = A.astype(np.complex64), B.astype(np.complex64)
    ia = ma if ma is not None else ([0] * PC if PA == 1 else list(range(PC)))
    ib = mb if mb is not None else ([0] * PC if PB == 1 else list(range(PC)))
    ref = np.stack([A[ia[p]].astype(np.complex128) @ B[ib[p]].astype(np.complex128) for p in range(PC)])
    buf = torch.full((PC * M * N + 2,), float("nan"), dtype=torch.complex64, device="cuda")
    c = buf[shift:shift + PC * M * N].view(PC, M, N)
    tn.tn_gemm_c64(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), c, engine=engine, map_a=ma, map_b=mb)
    got = c.cpu().numpy().astype(np.complex128)
    assert np.isfinite(got).all()
    tol = (2 * np.sqrt(K) + 4) * 2.0 ** -24
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
    rest = buf.cpu().numpy()
    assert np.isnan(rest[:shift]).all() and np.isnan(rest[shift + PC * M * N:]).all()   # nothing past the output


@pytest.mark.parametrize("shape", SHAPES, ids=[f"M{s[0]}N{s[1]}K{s[2]}P{s[3]}x{s[4]}x{s[5]}" for s in SHAPES])
def test_direct_kernel_bf16_products(tn, shape):
    """The BF16x3 engine on the direct kernel takes that engine's three products
    of bf16 parts: equal to them in FP64 up to FP32 rounding of three sums."""
    import torch
    M, N, K, PA, PB, PC, ma, mb = shape
    rng = np.random.default_rng(M * 7 + N * 3 + K + PA + 5 * PB + PC)
    A, B = (rng.normal(size=s) + 1j * rng.normal(size=s) for s in ((PA, M, K), (PB, K, N)))
    a, b = (torch.from_numpy(x.astype(np.complex64)) for x in (A, B))

    def parts(x):
        x = torch.view_as_real(x)
        hi = x.to(torch.bfloat16).to(torch.float32)
        lo = (x - hi).to(torch.bfloat16).to(torch.float32)
        return [torch.view_as_complex(y.contiguous()).to(torch.complex128).numpy() for y in (hi, lo)]

    (ah, al), (bh, bl) = parts(a), parts(b)
    ia = ma if ma is not None else ([0] * PC if PA == 1 else list(range(PC)))
    ib = mb if mb is not None else ([0] * PC if PB == 1 else list(range(PC)))
    if K == 2:                      # tf32 steps in every engine: plain products here
        ah, bh, al, bl = a.numpy().astype(np.complex128), b.numpy().astype(np.complex128), 0 * al, 0 * bl
    ref = np.stack([ah[i] @ bh[j] + ah[i] @ bl[j] + al[i] @ bh[j] for i, j in zip(ia, ib)])
    c = torch.full((PC, M, N), float("nan"), dtype=torch.complex64, device="cuda")
    tn.tn_gemm_c64(a.cuda(), b.cuda(), c, engine=3, map_a=ma, map_b=mb)
    got = c.cpu().numpy().astype(np.complex128)
    tol = 2 * (2 * np.sqrt(K) + 4) * 2.0 ** -24
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("engine", [1, 3, 4], ids=["tf32x3", "bf16x3", "fp16x3"])
@pytest.mark.parametrize("shape", [(512, 64, 256, 5), (256, 32, 128, 7), (512, 16, 64, 9), (256, 8, 32, 20),
                                   (256, 128, 64, 1), (4096, 1, 64, 53), (256, 2, 16, 70), (512, 4, 128, 33),
                                   (64, 1, 4, 3), (128, 4, 8, 200), (4096, 1024, 32, 1), (8192, 512, 4, 1),
                                   (2048, 64, 32, 24)], ids=str)
def test_gemm_kernels_on_request(tn, engine, shape):
    """pair = 1 keeps small shapes on the GEMM kernels: folded CTA-pair tiles, and
    narrow patterns as the columns of one matrix (ragged last tiles), and enough
    256 x 256 tiles for CTA pairs in tf32 too."""
    import torch
    M, N, K, P = shape
    rng = np.random.default_rng(M + N + K + P)
    A, B = ((rng.normal(size=s) + 1j * rng.normal(size=s)).astype(np.complex64) for s in ((1, M, K), (P, K, N)))
    ref = A.astype(np.complex128) @ B.astype(np.complex128)
    c = torch.full((P, M, N), float("nan"), dtype=torch.complex64, device="cuda")
    tn.tn_gemm_c64(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), c, engine=engine, pair=1)
    got = c.cpu().numpy()
    assert np.linalg.norm(got - ref) <= (1e-4 if engine == 3 else 1e-5) * np.linalg.norm(ref)


@pytest.mark.parametrize("engine", [1, 2, 3, 4], ids=["tf32x3", "simt", "bf16x3", "fp16x3"])
@pytest.mark.parametrize("shape", [(1, 4, 2, 3), (2, 64, 4, 3), (64, 8, 32, 5), (128, 32, 64, 2), (256, 64, 1024, 1)],
                         ids=str)
def test_operand_preparation_at_8_byte_starts(tn, engine, shape):
    """Operands that start on 8 but not on 16 bytes, and element counts that no
    16-byte load divides; two calls in a row with a larger one between them
    (the scratch is kept between calls)."""
    import torch
    M, N, K, P = shape
    rng = np.random.default_rng(M + N + K + P)
    A, B = ((rng.normal(size=s) + 1j * rng.normal(size=s)).astype(np.complex64) for s in ((P, M, K), (P, K, N)))
    ref = A.astype(np.complex128) @ B.astype(np.complex128)
    dev = []
    for X in (A, B):
        buf = torch.zeros(X.size + 1, dtype=torch.complex64, device="cuda")
        dev.append(buf[1:].view(X.shape))
        dev[-1].copy_(torch.from_numpy(X))
    c = torch.full((P, M, N), float("nan"), dtype=torch.complex64, device="cuda")
    big = [torch.ones(s, dtype=torch.complex64, device="cuda") for s in ((1, 512, 512), (1, 512, 512), (1, 512, 512))]
    for _ in range(2):
        c.fill_(float("nan"))
        tn.tn_gemm_c64(dev[0], dev[1], c, engine=engine, pair=1)
        got = c.cpu().numpy()
        assert np.linalg.norm(got - ref) <= (1e-4 if engine == 3 else 1e-5) * np.linalg.norm(ref)
        tn.tn_gemm_c64(*big, engine=engine, pair=1)
        assert float((big[2] - 512).abs().max()) <= 512 * (1e-4 if engine == 3 else 1e-5)
