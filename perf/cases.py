"""What this framework is used for, as cases that can be timed and compared.

Five kinds of work, all through the package's public calls:

* ``contract``   one circuit: reset the head, contract its kept slices, look the
                 amplitudes of the whole sparse state up (complex64);
* ``batch``      many small circuits contracted as one batch, then looked up;
* ``gemm``       one complex64 GEMM step of a contraction on its own;
* ``amplitudes`` a request's bitstrings looked up in a finished head;
* ``finish``     what follows a contraction: norms of the groups, one draw of
                 samples, linear and logarithmic XEB of those samples.

``listed()`` holds the sizes of the repository's own workloads and tests,
``draw()`` more of the same ranges.  Inputs come from the seed alone: the gates'
angles and kinds, the tails and the heads change with it, the sizes do not.
"""
import math

import numpy as np
import torch

import paper_2111_03011_gb300 as tn

ENGINES = {"auto": tn.TN_GEMM_AUTO, "fp16x3": tn.TN_GEMM_TC_FP16X3, "bf16x3": tn.TN_GEMM_TC_BF16X3}
METHODS = {"exact": tn.TN_SAMPLE_EXACT, "metropolis": tn.TN_SAMPLE_METROPOLIS, "frugal": tn.TN_SAMPLE_FRUGAL}
SEQUENCE = "ABCDCDAB"
EULER_GAMMA = 0.57721566490153286


# ------------------------------------------------------------------- cases

def _contract(name, rows, cols, cycles, n_open, tails, cuts, kept, engine, graph, trials=64, cap=28, auto_slice=0):
    return dict(name=name, kind="contract", rows=rows, cols=cols, cycles=cycles, n_open=n_open, tails=tails, cuts=cuts,
                kept=kept, engine=engine, graph=graph, trials=trials, cap=cap, auto_slice=auto_slice)


def listed():
    return [
        # the smallest sliced circuit of the parity tests: every slice's tensors
        # are a few thousand elements, so launches and latency are the whole cost
        _contract("contract_16q", 4, 4, 8, 6, 8, 2, 16, "auto", False),
        # a circuit of the serving mix, unsliced, on the default engine: a cold
        # start of the server contracts exactly this before it can answer
        _contract("contract_24q", 4, 6, 10, 7, 128, 0, 1, "auto", False),
        # the largest shape of the serving mix, sliced, on the fast engine; the
        # tail count is one that no power of two divides
        _contract("contract_25q", 5, 5, 12, 6, 99, 1, 4, "fp16x3", False),
        # the headline workload: 30 qubits, 14 cycles, 64 groups of 1,024; two of
        # its 64 slices as a captured graph (every slice has the same launches)
        _contract("contract_30q", 5, 6, 14, 10, 64, 3, 2, "fp16x3", True, trials=2048, cap=30),
        # the 40-qubit precision workload at a depth whose slice fits in a pass:
        # one of 1,024 slices, one tail, 2^12 amplitudes, the 1e-4 engine
        _contract("contract_40q", 5, 8, 12, 12, 1, 5, 1, "bf16x3", False, trials=512, cap=32, auto_slice=24),
        # the 53-qubit Sycamore lattice (rows = 0), 1,024 groups of 64, at the
        # depth that needs no automatic slicing: the many-pattern steps rule
        _contract("contract_53q", 0, 0, 7, 6, 1024, 0, 1, "auto", False, trials=512, cap=30, auto_slice=16),
        # many small circuits at once, the batched form
        dict(name="batch_12", kind="batch", circuits=12, n_open=6, tails=16, engine="fp16x3"),
        # one many-pattern step of the 30-qubit plan as a call of its own: short
        # K, gathered operands, an odd number of patterns
        dict(name="gemm_patterns", kind="gemm", M=512, N=64, K=8, PA=16, PB=8, PC=51, engine="auto"),
        # a stem step: long K, the matrix units are the bound
        dict(name="gemm_stem", kind="gemm", M=8192, N=1024, K=2048, PA=1, PB=1, PC=1, engine="fp16x3"),
        # an amplitude request as the benchmark's end-to-end step makes it:
        # pinned host bitstrings in, complex128 amplitudes out
        dict(name="amplitudes_host", kind="amplitudes", qubits=30, n_open=10, tails=64, n=65536, dtype="c128",
             where="host"),
        # the end of a serving run: 10^4 samples from few wide groups
        dict(name="finish_wide", kind="finish", qubits=30, n_open=10, tails=64, n=10000, method="exact",
             fidelity=0.0),
        # the paper's sampling: one sample from each of many groups of 64
        dict(name="finish_groups", kind="finish", qubits=53, n_open=6, tails=65536, n=65536, method="exact",
             fidelity=0.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["contract", "contract", "contract", "batch", "gemm", "gemm", "amplitudes", "finish"])
    if kind == "contract":
        rows, cols = rng.choice([(4, 4), (3, 6), (4, 5), (3, 7), (4, 6), (5, 5)])
        cuts = rng.randint(0, 2)
        # a prefix of the slices: fewer of them where a slice is large
        most = 4 ** cuts if rows * cols <= 20 else min(4, 4 ** cuts)
        c = _contract("", rows, cols, rng.randint(8, 12), rng.randint(6, 8), _log(rng, 12, 256), cuts,
                      2 ** rng.randint(0, most.bit_length() - 1), rng.choice(sorted(ENGINES)), rng.random() < 0.4)
        del c["name"]
        return c
    if kind == "batch":
        return dict(kind=kind, circuits=rng.randint(3, 12), n_open=rng.randint(5, 7), tails=_log(rng, 8, 64),
                    engine=rng.choice(["auto", "fp16x3"]))
    if kind == "gemm":
        while True:
            m, n, k = rng.randint(6, 14), rng.randint(2, 10), rng.randint(1, 11)
            p = _log(rng, 1, 64)
            big = p * 2 ** (max(m + k, k + n, m + n))
            if m + n + k + math.log2(p) <= 34 and big <= 2 ** 26:
                break
        pa, pb = rng.choice([(1, p), (p, 1), (p, p), (max(1, p // 3), max(1, p // 2))])
        return dict(kind=kind, M=2 ** m, N=2 ** n, K=2 ** k, PA=pa, PB=pb, PC=p, engine=rng.choice(sorted(ENGINES)))
    h = rng.randint(4, 12)
    tails = _log(rng, 1, 2 ** min(16, 20 - h))
    qubits = rng.randint(max(30, h + 17), 53)
    if kind == "amplitudes":
        return dict(kind=kind, qubits=qubits, n_open=h, tails=tails, n=_log(rng, 1000, 100000),
                    dtype=rng.choice(["c64", "c128"]), where=rng.choice(["host", "device"]))
    return dict(kind=kind, qubits=qubits, n_open=h, tails=tails, n=_log(rng, 100, 10000),
                method=rng.choice(["exact", "exact", "metropolis", "frugal"]), fidelity=rng.choice([0.0, 0.0, 0.4]))


# -------------------------------------------------------- circuits of the seed

class _Gate:
    def __init__(self, q0, q1, U):
        self.arity, self.q0, self.q1, self.U = (1 if q1 < 0 else 2), q0, q1, U


class _Circuit:
    def __init__(self, n_qubits, gates, first):
        self.n_qubits, self.gates, self.first = n_qubits, gates, first


def _couplers(rows, cols):
    """Number of qubits and the four coupler patterns: of a grid, or (rows = 0)
    of the 53-qubit staggered lattice."""
    pats = {c: [] for c in "ABCD"}
    if rows:
        for r in range(rows):
            for c in range(cols):
                if c + 1 < cols:
                    pats["AB"[c % 2]].append((r * cols + c, r * cols + c + 1))
                if r + 1 < rows:
                    pats["CD"[r % 2]].append((r * cols + c, (r + 1) * cols + c))
        return rows * cols, pats
    sites = [(r, c) for r in range(9) for c in range(6) if (r, c) != (8, 5)]
    at = {s: i for i, s in enumerate(sites)}
    for r, c in sites:
        for right, dc in ((True, r % 2), (False, r % 2 - 1)):
            if (r + 1, c + dc) in at:
                pats[("A" if right else "C") if r % 2 == 0 else ("B" if right else "D")].append(
                    (at[(r, c)], at[(r + 1, c + dc)]))
    return len(sites), pats


def _circuit(rows, cols, cycles, rng):
    """Layers of random square roots of X, Y and W with a layer of fSim gates after each, and a last
    layer of single-qubit gates."""
    n, pats = _couplers(rows, cols)
    x = np.array([[0, 1], [1, 0]], dtype=np.complex128)
    y = np.array([[0, -1j], [1j, 0]], dtype=np.complex128)
    roots = [(np.eye(2) - 1j * g) / math.sqrt(2) for g in (x, y, (x + y) / math.sqrt(2))]
    angle = {p: (math.pi / 2 + rng.uniform(-0.11, 0.11), math.pi / 6 + rng.uniform(-0.05, 0.05))
             for k in "ABCD" for p in pats[k]}
    gates, first, last = [], [], [-1] * n

    def singles():
        for q in range(n):
            k = int(rng.integers(3 if last[q] < 0 else 2))
            k += last[q] >= 0 and k >= last[q]
            last[q] = k
            gates.append(_Gate(q, -1, roots[k]))

    for t in range(cycles):
        singles()
        first.append(len(gates))
        for p in pats[SEQUENCE[t % 8]]:
            th, ph = angle[p]
            u = np.diag([1, math.cos(th), math.cos(th), np.exp(-1j * ph)]).astype(np.complex128)
            u[1, 2] = u[2, 1] = -1j * math.sin(th)
            gates.append(_Gate(p[0], p[1], u))
    singles()
    return _Circuit(n, gates, first)


def _tails(n_qubits, n_open, count, rng):
    """Distinct bitstrings over the qubits below the open ones (which are the last)."""
    got = set()
    while len(got) < count:
        got.update(int(v) for v in rng.integers(0, 1 << (n_qubits - n_open), size=count - len(got), dtype=np.uint64))
    return rng.permutation(np.array(sorted(got), dtype=np.uint64))


def _instance(case, seed):
    """Circuit, open qubits, tails and sliced edges of a contraction."""
    rng = np.random.default_rng([seed, 1])
    circ = _circuit(case["rows"], case["cols"], case["cycles"], rng)
    n, h = circ.n_qubits, case["n_open"]
    tails = _tails(n, h, case["tails"], rng)
    edges = []
    if case["cuts"]:                       # both inputs of gates spread over the middle cycle's layer
        mid = case["cycles"] // 2
        end = circ.first[mid + 1] if mid + 1 < len(circ.first) else len(circ.gates)
        layer = [i for i in range(circ.first[mid], end) if circ.gates[i].arity == 2]
        for j in np.linspace(0, len(layer) - 1, case["cuts"]).round().astype(int):
            edges += [(layer[j], 0, tn.TN_EDGE_SLICE, 0), (layer[j], 1, tn.TN_EDGE_SLICE, 0)]
    return circ, list(range(n - h, n)), tails, edges


def _batch_cases(case, seed):
    rng = np.random.default_rng([seed, 2, 0])
    shape = np.random.default_rng([case["circuits"], 3])     # the sizes are the case's, not the seed's
    grids = [(4, 4), (3, 6), (4, 5), (3, 7), (4, 6)]
    out = []
    for _ in range(case["circuits"]):
        r, c = grids[int(shape.integers(len(grids)))]
        out.append((dict(rows=r, cols=c, cycles=int(shape.integers(8, 13)), n_open=case["n_open"],
                         tails=case["tails"], cuts=0), int(rng.integers(1 << 31))))
    return out


def _bits(open_first, n_open, tails):
    """Every bitstring of the sparse state, group by group."""
    mu = np.arange(1 << n_open, dtype=np.uint64) << np.uint64(open_first)
    return (tails[:, None] | mu[None, :]).reshape(-1)


# ------------------------------------------------------------------ prepare

def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _contraction(case, seed, engine, **opts):
    circ, open_qubits, tails, edges = _instance(case, seed)
    plan = tn.tn_plan(circ, open_qubits, tails, edges, gemm=ENGINES[engine], **opts)
    head = tn.tn_head_create(plan)
    bits = _cuda(_bits(open_qubits[0], len(open_qubits), tails).view(np.int64))
    return dict(plan=plan, head=head, bits=bits, out=torch.empty(bits.numel(), dtype=torch.complex64, device="cuda"))


def _gemm_maps(case, rng):
    maps = []
    for p in (case["PA"], case["PB"]):
        maps.append(None if p in (1, case["PC"]) else [int(v) for v in rng.integers(0, p, case["PC"])])
    return maps


def _finished_head(case, seed):
    """A plan with the wanted sparse state and a head that holds Porter-Thomas amplitudes, as an earlier
    contraction (or a file) left them."""
    rng = np.random.default_rng([seed, 4])
    n, h = case["qubits"], case["n_open"]
    tails = _tails(n, h, case["tails"], rng)
    root = np.array([[1, -1j], [-1j, 1]]) / math.sqrt(2)
    circ = _Circuit(n, [_Gate(q, -1, root) for q in range(n)], [])
    plan = tn.tn_plan(circ, list(range(n - h, n)), tails)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    values = torch.randn((case["tails"], 1 << h, 2), dtype=torch.float64, device="cuda", generator=gen)
    values = torch.view_as_complex(values * 2.0 ** (-(n + 1) / 2))
    buf = torch.empty_like(values)
    head = tn.tn_head_create(plan, buf)
    buf.copy_(values)
    tn.tn_head_set_fidelity(head, 1.0)
    return plan, head, buf, tails, rng


def prepare(case, seed):
    kind = case["kind"]
    if kind == "contract":
        s = _contraction(case, seed, case["engine"], order_trials=case["trials"], max_log2_elements=case["cap"],
                         auto_slice=case["auto_slice"])
        return dict(s, kind=kind, kept=case["kept"], graph=case["graph"])
    if kind == "batch":
        items = [_contraction(c, sd, case["engine"]) for c, sd in _batch_cases(case, seed)]
        return dict(kind=kind, items=items)
    if kind == "gemm":
        rng = np.random.default_rng([seed, 5])
        gen = torch.Generator(device="cuda").manual_seed(seed)
        a, b = (torch.view_as_complex(torch.randn(s + (2,), device="cuda", generator=gen) / math.sqrt(2 * case["K"]))
                for s in ((case["PA"], case["M"], case["K"]), (case["PB"], case["K"], case["N"])))
        ma, mb = _gemm_maps(case, rng)
        c = torch.empty((case["PC"], case["M"], case["N"]), dtype=torch.complex64, device="cuda")
        return dict(kind=kind, a=a, b=b, c=c, map_a=ma, map_b=mb, engine=ENGINES[case["engine"]])
    plan, head, buf, tails, rng = _finished_head(case, seed)
    s = dict(kind=kind, plan=plan, head=head, buf=buf)
    if kind == "amplitudes":
        h, n = case["n_open"], case["n"]
        bits = tails[rng.integers(0, len(tails), n)] | (rng.integers(0, 1 << h, n, dtype=np.uint64) << np.uint64(case["qubits"] - h))
        bits = torch.from_numpy(bits.view(np.int64))
        wide = case["dtype"] == "c128"
        out = torch.empty(n, dtype=torch.complex128 if wide else torch.complex64)
        if case["where"] == "host":
            bits, out = bits.pin_memory(), out.pin_memory()
        else:
            bits, out = bits.cuda(), out.cuda()
        return dict(s, bits=bits, out=out, dtype=tn.TN_C128 if wide else tn.TN_C64)
    return dict(s, n=case["n"], method=METHODS[case["method"]], fidelity=case["fidelity"], seed=seed * 7919 + 11,
                out=torch.empty(case["n"], dtype=torch.int64, device="cuda"))


# ---------------------------------------------------------------------- run

def run(s):
    kind = s["kind"]
    if kind == "contract":
        tn.tn_head_reset(s["head"])
        (tn.tn_contract_slices_graph if s["graph"] else tn.tn_contract_slices)(s["plan"], 0, s["kept"], s["head"])
        return tn.tn_amplitudes(s["head"], s["bits"], out=s["out"], dtype=tn.TN_C64)
    if kind == "batch":
        items = s["items"]
        for x in items:
            tn.tn_head_reset(x["head"])
        tn.tn_contract_batch([x["plan"] for x in items], [(0, 1)] * len(items), [x["head"] for x in items])
        return [tn.tn_amplitudes(x["head"], x["bits"], out=x["out"], dtype=tn.TN_C64) for x in items]
    if kind == "gemm":
        return tn.tn_gemm_c64(s["a"], s["b"], s["c"], engine=s["engine"], map_a=s["map_a"], map_b=s["map_b"])
    if kind == "amplitudes":
        return tn.tn_amplitudes(s["head"], s["bits"], out=s["out"], dtype=s["dtype"])
    norm, groups = tn.tn_head_norm(s["head"], with_groups=True)
    samples = tn.tn_sample_ex(s["head"], s["n"], s["fidelity"], s["seed"], method=s["method"], out=s["out"])
    if s["fidelity"] > 0.0:                # uniform strings are mixed in: they are not all in the state
        return dict(norm=norm, groups=groups, samples=samples)
    linear, log_xeb = tn.tn_xeb(s["head"], samples)
    return dict(norm=norm, groups=groups, samples=samples, linear_xeb=linear, log_xeb=log_xeb)


# --------------------------------------------------------------------- work

def _macs(case, engine, seed=0, **opts):
    """Complex multiply-adds of one slice on the order that the planner finds, which is what a slice is counted by."""
    circ, open_qubits, tails, edges = _instance(case, seed)
    plan = tn.tn_plan(circ, open_qubits, tails, edges, gemm=ENGINES[engine], host_only=True, **opts)
    return tn.tn_plan_get_stats(plan)["tc_macs"]


def work(case):
    kind = case["kind"]
    if kind == "contract":
        n_amp = case["tails"] << case["n_open"]
        macs = _macs(case, case["engine"], order_trials=case["trials"], max_log2_elements=case["cap"],
                     auto_slice=case["auto_slice"])
        return {"bytes": n_amp * (16 + 8 + 8), "flops": 8.0 * macs * case["kept"]}
    if kind == "batch":
        macs = sum(_macs(c, case["engine"]) for c, _ in _batch_cases(case, 0))
        return {"bytes": case["circuits"] * (case["tails"] << case["n_open"]) * (16 + 8 + 8), "flops": 8.0 * macs}
    if kind == "gemm":
        m, n, k = case["M"], case["N"], case["K"]
        return {"bytes": 8 * (case["PA"] * m * k + case["PB"] * k * n + case["PC"] * m * n),
                "flops": 8 * case["PC"] * m * n * k}
    size = case["tails"] << case["n_open"]
    if kind == "amplitudes":
        wide = 16 if case["dtype"] == "c128" else 8
        return {"bytes": case["n"] * (8 + 16 + wide), "flops": 0}
    # every amplitude is read for the norms; a draw reads its group, the XEB one amplitude of it
    groups = min(case["tails"], case["n"])
    read = groups << case["n_open"] if case["method"] != "metropolis" else case["n"]
    return {"bytes": size * 16 + case["tails"] * 8 + read * 16 + case["n"] * (8 + 16), "flops": 3 * size}


# -------------------------------------------------------------------- exact

def _state_amplitudes(case, seed, kept):
    """Amplitudes of the sparse state from a complex128 state vector: the kept prefix of the slices leaves the low
    slice bits summed (their wires whole) and fixes the others to 0 (a projector on the cut wire)."""
    circ, open_qubits, tails, edges = _instance(case, seed)
    n = circ.n_qubits
    cut = {(g, leg) for j, (g, leg, _, _) in enumerate(edges) if j >= kept.bit_length() - 1}
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1
    order = list(range(n))                 # order[i]: the qubit of axis i (axis 0 is the slowest)
    single = [np.eye(2, dtype=np.complex128) for _ in range(n)]

    def apply(qubits, u):
        nonlocal psi, order
        at = sorted(range(len(qubits)), key=lambda j: order.index(qubits[j]))
        axes = [order.index(qubits[j]) for j in at]
        k = len(qubits)
        u = u.reshape([2] * (2 * k)).transpose(list(at) + [k + j for j in at]).reshape(1 << k, 1 << k)
        shape, last = [], -1
        for a in axes:
            shape += [1 << (a - last - 1), 2]
            last = a
        shape.append(1 << (n - 1 - last))
        front = list(range(1, 2 * k, 2)) + list(range(0, 2 * k + 1, 2))
        psi = torch.from_numpy(np.ascontiguousarray(u)).cuda() @ psi.reshape(shape).permute(front).reshape(1 << k, -1)
        order = [qubits[j] for j in at] + [q for q in order if q not in qubits]

    for i, g in enumerate(circ.gates):
        if g.arity == 1:
            single[g.q0] = g.U @ single[g.q0]
            continue
        pair = (g.q0, g.q1)
        before = [np.diag([1.0, 0.0]) @ single[q] if (i, leg) in cut else single[q] for leg, q in enumerate(pair)]
        apply(list(pair), g.U @ np.kron(*before))
        for q in pair:
            single[q] = np.eye(2, dtype=np.complex128)
    for q in range(n):
        if not np.array_equal(single[q], np.eye(2)):
            apply([q], single[q])
    bits = _cuda(_bits(open_qubits[0], len(open_qubits), tails).view(np.int64))
    index = torch.zeros_like(bits)
    for i, q in enumerate(order):
        index |= ((bits >> q) & 1) << (n - 1 - i)
    return psi.reshape(-1)[index]


def exact(case, seed):
    kind = case["kind"]
    if kind == "contract":
        # a state vector of 40 or 53 qubits does not exist
        return _state_amplitudes(case, seed, case["kept"]) if 0 < case["rows"] * case["cols"] <= 30 else None
    if kind == "batch":
        return [_state_amplitudes(c, sd, 1) for c, sd in _batch_cases(case, seed)]
    if kind == "gemm":
        s = prepare(case, seed)
        a, b = s["a"].to(torch.complex128), s["b"].to(torch.complex128)
        pick = [s["map_a"] or [0] * case["PC"], s["map_b"] or [0] * case["PC"]]
        for j, p in enumerate((case["PA"], case["PB"])):
            if p == case["PC"]:
                pick[j] = range(p)
        return torch.stack([a[i] @ b[j] for i, j in zip(*pick)])
    s = prepare(case, seed)
    value, tails = s["buf"], None
    h, first = case["n_open"], case["qubits"] - case["n_open"]

    def look_up(bits):
        nonlocal tails
        if tails is None:
            rng = np.random.default_rng([seed, 4])
            tails = _tails(case["qubits"], h, case["tails"], rng)
        by = np.argsort(tails)
        group = by[np.searchsorted(tails[by], bits & np.uint64((1 << first) - 1))]
        return value[_cuda(group), _cuda((bits >> np.uint64(first)).astype(np.int64))]

    if kind == "amplitudes":
        return look_up(s["bits"].cpu().numpy().view(np.uint64))
    groups = (value.real.square() + value.imag.square()).sum(1)
    out = dict(norm=float(groups.sum()), groups=groups, samples=None)
    if case["fidelity"] > 0.0:
        return out
    # the samples are whole numbers and have no 64-bit value of their own; the
    # XEB is a function of them, so it has none either
    return dict(out, linear_xeb=None, log_xeb=None)
