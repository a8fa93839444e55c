"""Workloads of this library at the sizes users run it, for timing and comparison.

A case is a dict of plain values; its "kind" says which public entry points one pass calls:

* circuit   a whole random Sycamore-pattern circuit from |0..0>: sim_reset or sim_front_run, then
            sim_apply_plan, amplitudes back in logical order; in FP32 followed by sim_reduce_async
* sliced    the same through the phases of a resident state with sliced qubits (sim_run_phases)
* block     one fused block on a random state (sim_apply_fused)
* permute   one qubit permutation of a random state (sim_permute)
* contract  the contraction of two tensors into a state (sim_contract)
* serve     a batch of small circuits through the server (srv_submit, srv_wait)

States are torch buffers handed to sim_create (ext_state), and every handle of a process orders
its work on one torch stream.  Streaming through pinned host memory is left out: its time is the
host link's, which other programs on the node share.
"""
import cmath
import math
import random

import numpy as np
import torch

import paper_1910_09534_gb300 as sim

PRECISIONS = {"fp32": sim.SIM_FP32, "fp16x3": sim.SIM_FP16X3, "fp16x3_tmem": sim.SIM_FP16X3_TMEM,
              "bf16x3": sim.SIM_BF16X3}


def listed():
    return [
        # the smallest whole run: the 3x4-grid, 8-cycle circuit, 4096 amplitudes, default arithmetic
        {"name": "circuit12_fp32", "kind": "circuit", "rows": 3, "n": 12, "cycles": 8, "precision": "fp32", "kmax": 4,
         "pairs": 0, "detuned": False},
        # a repeated medium circuit in split precision (the 4x5 grid at full depth)
        {"name": "circuit20_split", "kind": "circuit", "rows": 4, "n": 20, "cycles": 20, "precision": "fp16x3_tmem",
         "kmax": 5, "pairs": 0, "detuned": False},
        # the FP32 path of a serving-size circuit with its 2-bridging-gate front (4x6 grid)
        {"name": "circuit24_fp32", "kind": "circuit", "rows": 4, "n": 24, "cycles": 12, "precision": "fp32", "kmax": 4,
         "pairs": 2, "detuned": True},
        # the 30-qubit, 20-cycle run of the benchmark: contraction front, then blocks of <= 6 qubits
        {"name": "circuit30_split", "kind": "circuit", "rows": 5, "n": 30, "cycles": 20, "precision": "fp16x3_tmem",
         "kmax": 6, "pairs": 5, "detuned": False},
        # the 4x7 sub-lattice of the 33-qubit configuration through its sliced phases
        {"name": "sliced28_split", "kind": "sliced", "rows": 4, "n": 28, "cycles": 20, "precision": "fp16x3_tmem",
         "kmax": 6, "slice_bits": 3, "detuned": False},
        # one 6-qubit block on the 8 GiB state, split precision, targets spread over the register
        {"name": "block30_k6_split", "kind": "block", "n": 30, "precision": "fp16x3_tmem",
         "targets": "23 2 14 28 9 19"},
        # the fused k = 5 block in the default arithmetic (CUDA cores), one low target
        {"name": "block28_k5_fp32", "kind": "block", "n": 28, "precision": "fp32", "targets": "3 11 25 7 18"},
        # the default planner width (k_max 4) in the default arithmetic on the 8 GiB state
        {"name": "block30_k4_fp32", "kind": "block", "n": 30, "precision": "fp32", "targets": "1 12 6 27"},
        # a caller's own block on a cache-resident state: targets in no order, two of them low
        {"name": "block22_k5_split", "kind": "block", "n": 22, "precision": "fp16x3_tmem", "targets": "17 0 9 3 12"},
        # an arbitrary re-layout of the register
        {"name": "permute29", "kind": "permute", "n": 29, "perm_seed": 29},
        # contraction deferral's GEMM at a serving size: uneven sides, 4 bridging gates
        {"name": "contract27_split", "kind": "contract", "n1": 14, "n2": 13, "pairs": 4, "precision": "fp16x3_tmem"},
        # a burst of the serving stream's small circuits (16 qubits and a little around)
        {"name": "serve_small", "kind": "serve", "count": 24, "n_lo": 14, "n_hi": 18, "cycles": 12},
    ]


def draw(rng):
    kind = rng.choice(["circuit", "circuit", "sliced", "block", "block", "block", "permute", "contract", "serve"])
    if kind == "circuit":
        precision = rng.choice(["fp32", "fp16x3_tmem", "fp16x3_tmem", "bf16x3"])
        n = rng.randint(12, 27 if precision == "fp32" else 29)
        pairs = 0
        if n >= 22 and rng.random() < 0.6:  # the sizes that the server starts with a contraction front
            pairs = rng.randint(1, 2) if precision == "fp32" else rng.randint(2, 5)
        return {"kind": kind, "rows": math.isqrt(n), "n": n, "cycles": rng.randint(8, 20), "precision": precision,
                "kmax": rng.randint(3, 5) if precision == "fp32" else rng.randint(5, 6), "pairs": pairs,
                "detuned": rng.random() < 0.5}
    if kind == "sliced":
        precision = rng.choice(["fp32", "fp16x3_tmem"])
        return {"kind": kind, "rows": 4, "n": rng.randint(20, 27 if precision == "fp32" else 29),
                "cycles": rng.randint(8, 20), "precision": precision, "kmax": 4 if precision == "fp32" else 6,
                "slice_bits": rng.randint(2, 4), "detuned": rng.random() < 0.5}
    if kind == "block":
        n, k = rng.randint(13, 30), rng.randint(2, 6)
        return {"kind": kind, "n": n, "precision": rng.choice(["fp32", "fp32", "fp16x3_tmem", "fp16x3_tmem", "bf16x3",
                                                               "fp16x3"]),
                "targets": " ".join(str(q) for q in rng.sample(range(n), k))}
    if kind == "permute":
        return {"kind": kind, "n": rng.randint(14, 30), "perm_seed": rng.randrange(1 << 20)}
    if kind == "contract":
        precision = rng.choice(["fp16x3_tmem", "fp16x3_tmem", "bf16x3", "fp32"])
        return {"kind": kind, "n1": rng.randint(8, 14), "n2": rng.randint(8, 14),
                "pairs": rng.randint(1, 2 if precision == "fp32" else 5), "precision": precision}
    lo = rng.randint(10, 17)
    return {"kind": kind, "count": rng.randint(8, 32), "n_lo": lo, "n_hi": min(18, lo + rng.randint(0, 4)),
            "cycles": rng.randint(8, 16)}


# ---- circuits ---------------------------------------------------------------------------------

def _circuit(rows, n, cycles, detuned, rng):
    """Gate records (kind, q0, q1, theta, phi, d+, d-, d-off) of a random circuit: per cycle a
    random single-qubit gate on every qubit (never the one before it) and fSim gates on the
    couplers of the pattern, patterns in the order ABCDCDAB, then a last single-qubit layer."""
    cols = -(-n // rows)
    gates, prev = [], [-1] * n

    def layer():
        for q in range(n):
            prev[q] = rng.choice([g for g in range(3) if g != prev[q]])
            gates.append((prev[q], q, -1, 0.0, 0.0, 0.0, 0.0, 0.0))

    for t in range(cycles):
        layer()
        pattern = "ABCDCDAB"[t % 8]
        for q in range(n):
            r, c = divmod(q, cols)
            if (r + c) % 2 != (pattern in "BD"):
                continue
            other = q + 1 if pattern in "AB" else q + cols
            if other >= n or (pattern in "AB" and c + 1 == cols):
                continue
            extra = (0.0,) * 5
            if detuned:  # every coupler and cycle with its own unitary
                extra = (rng.uniform(-0.1, 0.1), rng.uniform(-0.1, 0.1)) + tuple(
                    rng.uniform(-math.pi, math.pi) for _ in range(3))
            gates.append((3, q, other, math.pi / 2 + extra[0], math.pi / 6 + extra[1]) + extra[2:])
    layer()
    return gates


def _circuit_of(case, seed):
    return _circuit(case["rows"], case["n"], case["cycles"], case["detuned"], random.Random(seed))


def _serve_circuits(case, seed):
    rng = random.Random(seed)
    out = []
    for i in range(case["count"]):
        n = case["n_lo"] + i % (case["n_hi"] - case["n_lo"] + 1)
        out.append((n, _circuit(math.isqrt(n), n, case["cycles"], False, rng)))
    return out


# ---- states -----------------------------------------------------------------------------------

_STREAM = []


def _stream():
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0].cuda_stream


class State:
    """What a program keeps between passes; its handles are given back with it."""

    def __init__(self, case):
        self.case = case
        self.undo = []

    def keep(self, handle, destroy):
        self.undo.append((destroy, handle))
        return handle

    def __del__(self):
        for destroy, handle in reversed(self.undo):
            destroy(handle)

    def handle(self, n, buf, slice_bits=0):
        """A handle whose state is buf, with the content that buf has."""
        content = buf.clone()
        torch.cuda.synchronize()
        h = sim.sim_create(n, slice_bits, stream=_stream(), ext_state=buf.data_ptr(), ext_bytes=8 << n)
        self.keep(h, sim.sim_destroy)
        sim.sim_sync(h)  # sim_create wrote |0..0>
        buf.copy_(content)
        torch.cuda.synchronize()
        return h


def _random_tensor(n, gen):
    """2^n Gaussian amplitudes of norm one, the distribution of a deep random circuit's state."""
    v = torch.randn(2 << n, generator=gen, device="cuda", dtype=torch.float32)
    v /= torch.linalg.vector_norm(v)
    return torch.view_as_complex(v.view(-1, 2))


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _random_unitary(k, seed):
    gen = torch.Generator().manual_seed(seed)
    z = torch.randn(1 << k, 1 << k, 2, generator=gen, dtype=torch.float64)
    q, r = torch.linalg.qr(torch.view_as_complex(z))
    d = torch.diagonal(r)
    return q * (d / d.abs())


def _permutation(case):
    perm = list(range(case["n"]))
    random.Random(case["perm_seed"]).shuffle(perm)
    return perm


def _bridged(case):
    """A gate list whose `pairs` fSim gates bridge the first n1 qubits and the others."""
    n1, n2 = case["n1"], case["n2"]
    return [(3, j % n1, n1 + j % n2, math.pi / 2, math.pi / 6) for j in range(case["pairs"])]


def prepare(case, seed):
    s = State(case)
    kind = case["kind"]
    if kind == "serve":
        s.circuits = [(n, sim.gates_array(g)) for n, g in _serve_circuits(case, seed)]
        s.amps = torch.empty(sum(1 << n for n, _ in s.circuits), dtype=torch.complex64, pin_memory=True)
        s.results = np.zeros((len(s.circuits), 2))
        s.server = s.keep(sim.srv_create(hbm_budget=8 << 30), sim.srv_destroy)
        return s
    if kind == "contract":
        n1, n2, pairs = case["n1"], case["n2"], case["pairs"]
        s.split = s.keep(sim.sim_split_create(n1 + n2, sim.gates_array(_bridged(case)), [0] * n1 + [1] * n2),
                         sim.sim_split_destroy)
        gen = _generator(seed)
        s.bufs = [_random_tensor(m + 2 * pairs, gen) for m in (n1, n2)]
        s.psi = torch.zeros(1 << (n1 + n2), dtype=torch.complex64, device="cuda")
        s.tensors = []
        for t, m in enumerate((n1, n2)):
            s.tensors.append(s.handle(m + 2 * pairs, s.bufs[t]))
            perm = [0] * (m + 2 * pairs)  # each wire at its canonical place
            for p, w in enumerate(sim.sim_split_canonical(s.split, t)):
                perm[w] = p
            sim.sim_set_layout(s.tensors[t], perm)
        s.h = s.handle(n1 + n2, s.psi)
        return s
    n = case["n"]
    precision = PRECISIONS.get(case.get("precision"))
    if kind in ("block", "permute"):
        s.psi = _random_tensor(n, _generator(seed))
        s.h = s.handle(n, s.psi)
        if kind == "block":
            s.targets = [int(q) for q in case["targets"].split()]
            s.matrix = _random_unitary(len(s.targets), seed).numpy()
        else:
            s.perm = _permutation(case)
        return s
    gates = sim.gates_array(_circuit_of(case, seed))
    s.psi = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
    s.h = s.handle(n, s.psi, case.get("slice_bits", 0))
    s.result = torch.zeros(3, dtype=torch.float64, pin_memory=True)
    s.identity = list(range(n))
    if kind == "sliced":
        b = case["slice_bits"]
        s.phases = s.keep(sim.sim_phases_create(n, gates, b, range(b), range(n - b, n), kmax=case["kmax"],
                                                precision=precision), sim.sim_phases_destroy)
        s.layout = sim.sim_phases_layout(s.phases, n, resident=True)[0]
        return s
    s.front = None
    if case["pairs"]:
        side, front = sim.sim_split_choose(n, gates, case["pairs"])
        split = s.keep(sim.sim_split_create(n, gates[:front], side), sim.sim_split_destroy)
        s.front = s.keep(sim.sim_front_create(s.h, split, kmax=case["kmax"], precision=precision),
                         sim.sim_front_destroy)
        gates = gates[front:]
    s.plan = s.keep(sim.sim_plan_create(n, gates, kmax=case["kmax"], precision=precision), sim.sim_plan_destroy)
    s.layout = None
    if s.front is not None:
        s.layout = sim.sim_plan_layout_front(s.plan, split, n)[0]
    elif n > 20:  # as the server does
        s.layout = sim.sim_plan_layout(s.plan, n)[0]
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "serve":
        amps, at, tickets = s.amps.numpy(), 0, []
        for n, gates in s.circuits:
            tickets.append(sim.srv_submit(s.server, n, gates, amps[at:at + (1 << n)]))
            at += 1 << n
        for i, t in enumerate(tickets):
            s.results[i] = sim.srv_wait(s.server, t)[:2]
        return s.amps, s.results
    if kind == "contract":
        sim.sim_contract(s.h, s.tensors[0], s.tensors[1], s.split, PRECISIONS[case["precision"]])
        return s.psi
    if kind == "block":
        sim.sim_apply_fused(s.h, s.targets, s.matrix, PRECISIONS[case["precision"]])
        return s.psi
    if kind == "permute":
        # the caller names the new places of the qubits; the labels stay as they were
        sim.sim_permute(s.h, s.perm)
        sim.sim_set_layout(s.h, range(case["n"]))
        return s.psi
    if s.layout is not None:
        sim.sim_set_layout(s.h, s.layout)
    if kind == "sliced":
        sim.sim_reset(s.h)
        sim.sim_run_phases(s.h, s.phases)
    else:
        if s.front is not None:
            sim.sim_front_run(s.h, s.front)
        else:
            sim.sim_reset(s.h)
        sim.sim_apply_plan(s.h, s.plan)
    if s.layout is not None:
        sim.sim_permute(s.h, s.identity)
    if case["precision"] != "fp32":
        return s.psi
    sim.sim_reduce_async(s.h, s.result.numpy())
    return s.psi, s.result


def work(case):
    kind = case["kind"]
    if kind == "block":
        k = len(case["targets"].split())
        return {"bytes": 16.0 * 2 ** case["n"], "flops": 8.0 * 2 ** (case["n"] + k)}
    if kind == "permute":
        return {"bytes": 16.0 * 2 ** case["n"], "flops": 0.0}
    if kind == "contract":
        n1, n2, e = case["n1"], case["n2"], 2 * case["pairs"]
        return {"bytes": 8.0 * (2 ** (n1 + e) + 2 ** (n2 + e) + 2 ** (n1 + n2)), "flops": 8.0 * 2 ** (n1 + n2 + e)}
    circuits = _serve_circuits(case, 0) if kind == "serve" else [(case["n"], _circuit_of(case, 0))]
    # every amplitude written once; each two-qubit gate (the single-qubit ones folded in) as 4x4 products
    return {"bytes": float(sum(8 << n for n, _ in circuits)),
            "flops": float(sum(32 * sum(g[0] == 3 for g in gates) << n for n, gates in circuits))}


# ---- the same in 64 bits, gate by gate --------------------------------------------------------

def _gate_1q(kind):
    x = torch.tensor([[0, 1], [1, 0]], dtype=torch.complex128)
    y = torch.tensor([[0, -1j], [1j, 0]], dtype=torch.complex128)
    p = (x, y, (x + y) / math.sqrt(2))[kind]
    return (torch.eye(2, dtype=torch.complex128) - 1j * p) / math.sqrt(2)


def _gate_fsim(theta, phi, dplus=0.0, dminus=0.0, dminus_off=0.0):
    """Eq. 1, index b(q0) + 2 b(q1)."""
    m = torch.zeros(4, 4, dtype=torch.complex128)
    c, s = math.cos(theta), math.sin(theta)
    m[0, 0] = 1
    m[1, 1] = cmath.exp(1j * (dplus + dminus)) * c
    m[1, 2] = -1j * cmath.exp(1j * (dplus - dminus_off)) * s
    m[2, 1] = -1j * cmath.exp(1j * (dplus + dminus_off)) * s
    m[2, 2] = cmath.exp(1j * (dplus - dminus)) * c
    m[3, 3] = cmath.exp(1j * (2 * dplus - phi))
    return m


def _on_pair(psi, a, b, m):
    """psi <- m psi on qubits a, b (index b(a) + 2 b(b) of m)."""
    lo, hi = min(a, b), max(a, b)
    if a > b:
        m = m[[0, 2, 1, 3]][:, [0, 2, 1, 3]]
    v = psi.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
    part = [v[:, j >> 1, :, j & 1, :] for j in range(4)]
    new = []
    for r in range(4):
        y = None
        for c in range(4):
            w = complex(m[r, c])
            if w != 0:
                y = part[c] * w if y is None else y.add_(part[c], alpha=w)
        new.append(y)
    for r in range(4):
        part[r].copy_(new[r])


def _run_64(n, gates):
    """The circuit's amplitudes, single-qubit gates folded into the two-qubit gate after them (the
    last ones into the gate before)."""
    eye = torch.eye(2, dtype=torch.complex128)
    pend, last, ops = [eye] * n, [None] * n, []
    for g in gates:
        if g[0] < 3:
            pend[g[1]] = _gate_1q(g[0]) @ pend[g[1]]
            continue
        a, b = g[1], g[2]
        ops.append([a, b, _gate_fsim(*g[3:]) @ torch.kron(pend[b], pend[a])])
        pend[a] = pend[b] = eye
        last[a] = last[b] = len(ops) - 1
    for q in range(n):
        if last[q] is None:
            ops.append([q, (q + 1) % n, torch.kron(eye, pend[q])])
            continue
        op = ops[last[q]]
        op[2] = (torch.kron(eye, pend[q]) if op[0] == q else torch.kron(pend[q], eye)) @ op[2]
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1
    for a, b, m in ops:
        _on_pair(psi, a, b, m)
    return psi


def _sums_64(psi):
    p = psi.real.square() + psi.imag.square()
    return float(p.sum()), float(p.square_().sum()) * psi.numel()


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        states = [_run_64(n, g) for n, g in _serve_circuits(case, seed)]
        return (torch.cat([x.cpu() for x in states]),
                torch.tensor([_sums_64(x) for x in states], dtype=torch.float64))
    if kind == "contract":
        gen = _generator(seed)
        t1, t2 = [_random_tensor(m + 2 * case["pairs"], gen).to(torch.complex128).view(-1, 1 << m)
                  for m in (case["n1"], case["n2"])]
        return (t2.t() @ t1).reshape(-1)
    if kind == "permute":
        n, perm = case["n"], _permutation(case)
        psi = _random_tensor(n, _generator(seed))
        out = torch.empty_like(psi)
        step = min(1 << n, 1 << 24)
        low = torch.arange(step, device="cuda")
        for first in range(0, 1 << n, step):
            index = first + low  # the place of bit perm[q] of the new index was q
            source = torch.zeros_like(index)
            for q, p in enumerate(perm):
                source |= ((index >> p) & 1) << q
            out[first:first + step] = psi[source]
        return out
    if kind == "block":
        n, targets = case["n"], [int(q) for q in case["targets"].split()]
        k = len(targets)
        m = _random_unitary(k, seed).to("cuda")
        psi = _random_tensor(n, _generator(seed))
        shape, axis_of, top = [], {}, n
        for q in sorted(targets, reverse=True):  # [rest, target, rest, target, ..]
            shape += [1 << (top - 1 - q), 2]
            axis_of[q] = len(shape) - 1
            top = q
        shape.append(1 << top)
        v = psi.view(shape)
        first = [axis_of[q] for q in reversed(targets)]  # bit j of the row index is targets[j]
        order = first + [i for i in range(len(shape)) if i not in first]
        x = v.permute(order).reshape(1 << k, -1)
        y = torch.empty_like(x, dtype=torch.complex128)
        for i in range(0, x.shape[1], 1 << 22):
            y[:, i:i + (1 << 22)] = m @ x[:, i:i + (1 << 22)].to(torch.complex128)
        back = [0] * len(order)
        for i, o in enumerate(order):
            back[o] = i
        return y.view([shape[o] for o in order]).permute(back).reshape(-1)
    psi = _run_64(case["n"], _circuit_of(case, seed))
    if case["precision"] != "fp32":
        return psi
    norm, s2 = _sums_64(psi)
    return psi, torch.tensor([norm, s2, s2 - 1], dtype=torch.float64)
