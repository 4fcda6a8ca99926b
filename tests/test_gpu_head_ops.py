"""Norms, XEB and the exact sampler on heads of every shape class (one member
to 2^13, fewer and more samples than groups), against NumPy.

The sampler's definition -- weights rounded operation by operation, prefix sums
by a 32-wide scan per chunk and one addition per chunk -- is repeated here in
FP64, so the draws must be equal bit for bit: also for groups with zeros and
repeated values, where FP32 estimates of the prefixes cannot decide, for
magnitudes outside the FP32 range, and for groups that are all zero."""
import math

import numpy as np
import pytest

import circuit_inputs as ci
import oracle as O

pytestmark = pytest.mark.gpu

NQ = 40


@pytest.fixture(scope="module")
def tn():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2111_03011_gb300 as m
    return m


def _head(tn, H):
    import torch
    L, l = H.shape
    h = l.bit_length() - 1
    oq = list(range(NQ - h, NQ))
    tails = ci.draw_tails(NQ, oq, L, seed=L + h)
    c = ci.make_grid_circuit(2, 2, 1, seed=1)
    c.n_qubits = NQ
    plan = tn.tn_plan(c, oq, tails, host_fold_log2=-1)
    buf = torch.zeros((L, l), dtype=torch.complex128, device="cuda")
    head = tn.tn_head_create(plan, buf)
    buf.copy_(torch.from_numpy(H))
    tn.tn_head_set_fidelity(head, 1.0)
    torch.cuda.synchronize()
    return plan, head, buf, tails, oq


def _values(kind, L, l, seed):
    rng = np.random.default_rng(seed)
    H = (rng.normal(size=(L, l)) + 1j * rng.normal(size=(L, l))) * 2.0 ** (-(NQ + 1) / 2)
    if kind == "ties":                          # zeros, equal members, all-zero groups
        H = np.where(rng.random((L, l)) < 0.6, 0.0, np.round(H * 2.0 ** 21) * 2.0 ** -21)
        H[::5] = 0.0
    elif kind == "tiny":
        H = H * 2.0 ** -300
    elif kind == "huge":
        H = H * 2.0 ** 200
    elif kind == "spread":
        H = H * 2.0 ** rng.integers(-60, 60, size=(L, l)).astype(np.float64)
    return H


def _reference(H, tails, oq, n, seed):
    L, l = H.shape
    out = np.zeros(n, dtype=np.uint64)
    prefix = {}
    for i in range(n):
        g = i % L
        r = O.philox4x32_10((i & 0xFFFFFFFF, i >> 32, 0, 0), (seed & 0xFFFFFFFF, seed >> 32))
        u = (((r[3] << 32) | r[2]) >> 11) * 2.0 ** -53
        if g not in prefix:
            w = H[g].real * H[g].real + H[g].imag * H[g].imag
            w = np.pad(w, (0, -l % 32)).reshape(-1, 32)
            for d in (1, 2, 4, 8, 16):
                w[:, d:] = w[:, d:] + w[:, :-d]
            carry, P = 0.0, np.empty_like(w)
            for c in range(w.shape[0]):
                P[c] = carry + w[c]
                carry = carry + w[c, 31]
            prefix[g] = (P.reshape(-1)[:l], carry)
        P, Z = prefix[g]
        if Z > 0.0:
            hit = np.nonzero(P > u * Z)[0]
            mu = int(hit[0]) if hit.size else l - 1
        else:
            mu = min(int(u * l), l - 1)
        out[i] = int(tails[g]) | sum(((mu >> j) & 1) << q for j, q in enumerate(oq))
    return out


SHAPES = [(7, 0, 20), (5, 3, 40), (9, 5, 50), (33, 6, 33), (33, 6, 200), (5, 7, 5), (5, 7, 64), (3, 8, 3),
          (2, 12, 300), (1, 13, 100), (400, 6, 380)]


@pytest.mark.parametrize("kind", ["plain", "ties", "tiny", "huge", "spread"])
@pytest.mark.parametrize("L,h,n", SHAPES)
def test_exact_draws_bit_for_bit(tn, L, h, n, kind):
    H = _values(kind, L, 1 << h, seed=L + 31 * h)
    plan, head, buf, tails, oq = _head(tn, H)
    seed = 0x9ABC_DEF0_1234
    assert np.array_equal(tn.tn_sample(head, n, 0.0, seed), _reference(H, tails, oq, n, seed))


@pytest.mark.parametrize("L,h", [(1, 0), (7, 2), (1000, 3), (333, 4), (65, 6), (3, 9), (40, 10), (2, 13), (1, 16), (9000, 1)])
def test_norms_and_xeb(tn, L, h):
    """FP64 sums of up to 2^16 terms in any order: within 2^16 units of 2^-53 of
    the sum of magnitudes, and far closer in fact."""
    H = _values("plain", L, 1 << h, seed=L * 7 + h)
    plan, head, buf, tails, oq = _head(tn, H)
    w = np.abs(H) ** 2
    N, Z = tn.tn_head_norm(head, with_groups=True)
    assert tn.tn_head_norm(head) == N
    assert np.allclose(Z, w.sum(axis=1), rtol=2.0 ** -42, atol=0) and math.isclose(N, w.sum(), rel_tol=2.0 ** -42)
    rng = np.random.default_rng(5)
    g, mu = rng.integers(0, L, 700), rng.integers(0, 1 << h, 700)
    bits = np.array([int(tails[a]) | sum(((int(b) >> j) & 1) << q for j, q in enumerate(oq)) for a, b in zip(g, mu)],
                    dtype=np.uint64)
    lin, log = tn.tn_xeb(head, bits)
    p = w[g, mu]
    scale = np.abs(np.log(p)).mean() + 100
    assert math.isclose(lin, 2.0 ** NQ * p.mean() - 1, rel_tol=2.0 ** -40, abs_tol=2.0 ** -40)
    assert abs(log - (NQ * math.log(2) + 0.57721566490153286 + np.log(p).mean())) <= 2.0 ** -40 * scale


@pytest.mark.parametrize("where", ["numpy", "pinned", "device"])
def test_amplitudes_from_any_memory(tn, where):
    import torch
    H = _values("plain", 12, 16, seed=3)
    plan, head, buf, tails, oq = _head(tn, H)
    bits = np.array([int(t) | (mu << (NQ - 4)) for t in tails for mu in range(16)], dtype=np.uint64)
    if where == "numpy":
        got = tn.tn_amplitudes(head, bits)
        s = tn.tn_sample(head, 30, 0.0, 9)
    else:
        b, o = torch.from_numpy(bits.view(np.int64)), torch.zeros(bits.size, dtype=torch.complex128)
        so = torch.zeros(30, dtype=torch.int64)
        b, o, so = (x.pin_memory() if where == "pinned" else x.cuda() for x in (b, o, so))
        got = tn.tn_amplitudes(head, b, out=o).cpu().numpy()
        s = tn.tn_sample(head, 30, 0.0, 9, out=so).cpu().numpy().view(np.uint64)
    assert np.array_equal(got.reshape(12, 16), H)
    assert np.array_equal(s, _reference(H, tails, oq, 30, 9))
    if where != "numpy":
        b[5] = int(bits[5]) ^ 1
        b[9] = int(bits[9]) ^ 2
        missing = [i for i in (5, 9) if int(b[i].item()) & ((1 << (NQ - 4)) - 1) not in [int(t) for t in tails]]
        with pytest.raises(tn.TNError) as e:
            tn.tn_amplitudes(head, b, out=o)
        assert e.value.code == tn.TN_ERR_NOT_IN_STATE and f"bitstring {missing[0]} " in str(e.value)
        assert o.cpu().numpy()[missing[0]] == 0


def test_open_qubits_that_are_not_consecutive(tn):
    import torch
    oq = [5, 2, 39, 17]
    L, h = 9, 4
    H = _values("plain", L, 1 << h, seed=8)
    tails = ci.draw_tails(NQ, oq, L, seed=4)
    c = ci.make_grid_circuit(2, 2, 1, seed=1)
    c.n_qubits = NQ
    plan = tn.tn_plan(c, oq, tails, host_fold_log2=-1)
    buf = torch.zeros((L, 1 << h), dtype=torch.complex128, device="cuda")
    head = tn.tn_head_create(plan, buf)
    buf.copy_(torch.from_numpy(H))
    torch.cuda.synchronize()
    bits = np.array([int(t) | sum(((mu >> j) & 1) << q for j, q in enumerate(oq)) for t in tails
                     for mu in range(1 << h)], dtype=np.uint64)
    assert np.array_equal(tn.tn_amplitudes(head, bits).reshape(L, -1), H)
    lin, _ = tn.tn_xeb(head, bits)
    assert math.isclose(lin, 2.0 ** NQ * (np.abs(H) ** 2).mean() - 1, rel_tol=2.0 ** -40, abs_tol=2.0 ** -40)
    tn.tn_head_set_fidelity(head, 1.0)
    assert np.array_equal(tn.tn_sample(head, 40, 0.0, 3), _reference(H, tails, oq, 40, 3))
