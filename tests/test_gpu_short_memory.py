"""A plan on a device with room for one pass but not for the copies of its
batched steps: it is accepted, runs its passes one by one and gives the same
bits."""
import numpy as np
import pytest

import circuit_inputs as ci

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gemm", [1, 4])
def test_plan_without_room_for_batched_copies(gemm):
    import torch
    import paper_2111_03011_gb300 as tn
    cfg = ci.config_small(4, 6, 10, seed=4, n_open=7, L=256, n_cut_gates=3)
    args = (cfg["circuit"], cfg["open_qubits"], cfg["tails"], cfg["edges"])
    bits = np.array([int(t) | (mu << 17) for t in cfg["tails"] for mu in range(128)], dtype=np.uint64)

    def amplitudes(plan):
        head = tn.tn_head_create(plan)
        tn.tn_contract_slices(plan, 3, 30, head)
        return tn.tn_amplitudes(head, bits)

    plan = tn.tn_plan(*args, gemm=gemm)
    d = tn.tn_plan_describe(plan)
    most, stride = d["batch"]
    small = d["workspace_bytes"] - (most - 1) * stride
    assert most > 1 and (most - 1) * stride >= 48 << 20
    want = amplitudes(plan)
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    spare = small + (24 << 20)                 # the plan's tables and leaves, and the head, come on top
    fill = torch.empty(torch.cuda.mem_get_info()[0] - spare, dtype=torch.uint8, device="cuda")
    tight = tn.tn_plan(*args, gemm=gemm)
    got = amplitudes(tight)
    del fill
    torch.cuda.empty_cache()
    t = tn.tn_plan_describe(tight)
    assert t["batch"][0] == 1 and t["workspace_bytes"] == small
    assert np.array_equal(got, want)
