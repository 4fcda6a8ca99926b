"""Buffers that a caller hands in as they come: results and bitstrings in pinned
memory that starts on fewer bytes than a kernel moves at a time, and results
written over the bitstrings they belong to.

The rules that send such buffers through the staging buffer are checked on the
CPU (compiled from their header); on the GPU the values of the calls are."""
import os
import subprocess

import numpy as np
import pytest

import circuit_inputs as ci

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NQ, N_OPEN, GROUPS = 40, 4, 12

CHECK = r"""
#include "buffers.h"
#include <cstdio>
int main() {
  static_assert(sizeof(void*) == 8, "");
  char* b = (char*)0x100000;
  int bad = 0;
  for (int o = 0; o < 64; ++o) {
    bad += tn::kernel_aligned(b + o, 16) != (o % 16 == 0);   // complex128 results
    bad += tn::kernel_aligned(b + o, 8) != (o % 8 == 0);     // complex64 results, bitstrings, samples
  }
  // byte by byte against the definition
  for (int na = 0; na < 5; ++na)
    for (int nb = 0; nb < 5; ++nb)
      for (int d = -6; d <= 6; ++d) {
        bool want = false;
        for (int i = 0; i < na; ++i)
          for (int j = 0; j < nb; ++j) want |= i == d + j;
        bad += tn::ranges_overlap(b, na, b + d, nb) != want;
      }
  std::printf("%d\n", bad);
  return bad != 0;
}
"""


def test_rules_on_buffers(tmp_path):
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(CHECK)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2111_03011_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    assert subprocess.run([str(exe)], stdout=subprocess.PIPE, check=True).stdout == b"0\n"


@pytest.fixture(scope="module")
def head():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2111_03011_gb300 as tn
    rng = np.random.default_rng(7)
    H = (rng.normal(size=(GROUPS, 1 << N_OPEN)) + 1j * rng.normal(size=(GROUPS, 1 << N_OPEN))) * 2.0 ** -20
    oq = list(range(NQ - N_OPEN, NQ))
    tails = ci.draw_tails(NQ, oq, GROUPS, seed=3)
    c = ci.make_grid_circuit(2, 2, 1, seed=1)
    c.n_qubits = NQ
    plan = tn.tn_plan(c, oq, tails, host_fold_log2=-1)
    buf = torch.zeros(H.shape, dtype=torch.complex128, device="cuda")
    h = tn.tn_head_create(plan, buf)
    buf.copy_(torch.from_numpy(H))
    tn.tn_head_set_fidelity(h, 1.0)
    torch.cuda.synchronize()
    bits = np.array([int(t) | (mu << (NQ - N_OPEN)) for t in tails for mu in range(1 << N_OPEN)], dtype=np.uint64)
    return tn, h, H.reshape(-1), bits, (plan, buf)


def _block(where, nbytes):
    """A byte buffer on a 256-byte boundary."""
    import torch
    t = torch.zeros(nbytes + 256, dtype=torch.uint8)
    t = t.pin_memory() if where == "pinned" else t.cuda() if where == "device" else t
    o = -t.data_ptr() % 256
    return t[o:o + nbytes]


class _At:
    """What the binding wants of a buffer: its address and element count."""

    def __init__(self, block, offset, count):
        self.block, self.address, self.count = block, block.data_ptr() + offset, count

    def data_ptr(self):
        return self.address

    def numel(self):
        return self.count


def _put(block, offset, a):
    import torch
    block[offset:offset + a.nbytes] = torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1))


def _get(block, offset, n, dtype):
    raw = block[offset:offset + n * np.dtype(dtype).itemsize].cpu().numpy()
    return np.frombuffer(raw.tobytes(), dtype=dtype)


@pytest.mark.gpu
@pytest.mark.parametrize("where", ["pinned", "device", "pageable"])
@pytest.mark.parametrize("wide", [True, False], ids=["c128", "c64"])
@pytest.mark.parametrize("at_in,at_out", [(0, 0), (0, 8), (4, 4), (1, 3)])
def test_results_and_bitstrings_at_any_alignment(head, where, wide, at_in, at_out):
    tn, h, H, bits, _ = head
    n, t = bits.size, np.complex128 if wide else np.complex64
    src, dst = _block(where, n * 8 + 64), _block(where, n * 16 + 64)
    _put(src, at_in, bits)
    tn.tn_amplitudes(h, _At(src, at_in, n), out=_At(dst, at_out, n), dtype=tn.TN_C128 if wide else tn.TN_C64)
    assert np.array_equal(_get(dst, at_out, n, t), H.astype(t))
    assert not _get(dst, 0, at_out, np.uint8).any()
    end = at_out + n * np.dtype(t).itemsize
    assert not dst[end:].cpu().numpy().any()
    # the same buffers as samples: what XEB reads and a draw writes
    want = tn.tn_xeb(h, bits)
    assert tn.tn_xeb(h, _At(src, at_in, n)) == want
    tn.tn_sample(h, n, 0.0, 9, out=_At(src, at_in, n))
    assert np.array_equal(_get(src, at_in, n, np.uint64), tn.tn_sample(h, n, 0.0, 9))


@pytest.mark.gpu
@pytest.mark.parametrize("where", ["pinned", "device", "pageable"])
@pytest.mark.parametrize("wide", [True, False], ids=["c128", "c64"])
@pytest.mark.parametrize("shift", [0, 8, 512])
def test_results_over_the_bitstrings(head, where, wide, shift):
    tn, h, H, bits, _ = head
    n, t = 50 * bits.size, np.complex128 if wide else np.complex64
    block = _block(where, n * 16 + 1024)
    pick = np.random.default_rng(2).integers(0, bits.size, n)
    _put(block, shift, bits[pick])
    tn.tn_amplitudes(h, _At(block, shift, n), out=_At(block, 0, n), dtype=tn.TN_C128 if wide else tn.TN_C64)
    assert np.array_equal(_get(block, 0, n, t), H[pick].astype(t))
