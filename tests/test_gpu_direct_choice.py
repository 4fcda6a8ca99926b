"""The shapes of test_gpu_direct.py do run on the direct kernel: with pair = 1
the same call runs on the GEMM kernels, which round differently, and either
call repeats its own bits.  (BF16x3, where the direct kernel takes three products
for one, runs the larger of them on the GEMM.)"""
import numpy as np
import pytest

from test_gpu_direct import SHAPES

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", [1, 4], ids=["tf32x3", "fp16x3"])
def test_shapes_take_the_direct_kernel(engine):
    import torch
    import paper_2111_03011_gb300 as tn
    seen = 0
    for M, N, K, PA, PB, PC, ma, mb in SHAPES:
        if M * N * PC < 256 or K < 8:
            continue                            # too few roundings to tell the forms apart
        gen = torch.Generator(device="cuda").manual_seed(M + N + K + PC)
        a, b = (torch.view_as_complex(torch.randn(s + (2,), device="cuda", generator=gen))
                for s in ((PA, M, K), (PB, K, N)))
        out = []
        for pair in (0, 0, 1, 1):
            c = torch.empty((PC, M, N), dtype=torch.complex64, device="cuda")
            tn.tn_gemm_c64(a, b, c, engine=engine, map_a=ma, map_b=mb, pair=pair)
            out.append(c.cpu().numpy())
        assert np.array_equal(out[0], out[1]) and np.array_equal(out[2], out[3])
        assert not np.array_equal(out[0], out[2]), (M, N, K, PC)
        seen += 1
    assert seen >= 8
