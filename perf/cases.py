"""Performance cases of the state-vector engine: what they run, on which
inputs, and what they return.

A case is a dict of plain values.  ``prepare`` makes what a user's program
holds before the call (registers, gate lists, plans, batches), from the seed;
``run`` is one pass through the public calls of ``qudit.py``; ``work`` counts
the bytes and operations that the pass cannot do without; ``exact`` gives the
outputs in 64 bits from plain torch, without the engine.

Registers are written "2x8,4x11": eight qubits (the least significant digits)
followed by eleven ququarts.
"""
import math

import numpy as np
import torch

from paper_2211_07918_gb300 import costmodel, workloads
from paper_2211_07918_gb300 import qudit as qd

PLANS = {"none": qd.QD_PLAN_NONE, "greedy": qd.QD_PLAN_GREEDY, "exhaustive": qd.QD_PLAN_EXHAUSTIVE,
         "learned": qd.QD_PLAN_LEARNED}
PREC = {"c64": qd.QD_C64, "c128": qd.QD_C128}
DTYPE = {"c64": torch.complex64, "c128": torch.complex128}
SIZE = {"c64": 8, "c128": 16}


def dims_of(text):
    out = []
    for part in text.split(","):
        d, m = part.split("x")
        out += [int(d)] * int(m)
    return out


def text_of(dims):
    parts = []
    for d in dims:
        if parts and parts[-1][0] == d:
            parts[-1][1] += 1
        else:
            parts.append([d, 1])
    return ",".join("%dx%d" % (d, m) for d, m in parts)


# ------------------------------------------------------------------ cases

def listed():
    return [
        # the paper's own scale: a tiny hybrid register in double precision, its circuit built, run and
        # printed as kets in one go (latency of the calls, launches and host work)
        {"name": "small_ket_c128", "kind": "small", "dims": "3x4,2x2", "gates": 40, "prec": "c128"},
        # per-gate execution of a prepared circuit on a register that fits L2 (14 qutrits), both precisions
        {"name": "qutrits14_gates_c64", "kind": "circuit", "family": "qutrit", "dims": "3x14", "gates": 500,
         "plan": "none", "prec": "c64"},
        {"name": "qutrits14_gates_c128", "kind": "circuit", "family": "qutrit", "dims": "3x14", "gates": 300,
         "plan": "none", "prec": "c128"},
        # the flagship workload (Haar layer, ququart QFT, Toffoli ladder) with the learned fusion plan
        {"name": "qft_ladder_c64", "kind": "circuit", "family": "qft", "dims": "2x8,4x11", "gates": 0,
         "plan": "learned", "prec": "c64"},
        # a random circuit of every gate kind on odd strides (qutrits below qubits), fused
        {"name": "mixed_fused_c64", "kind": "circuit", "family": "mixed", "dims": "3x16,2x4", "gates": 60,
         "plan": "exhaustive", "prec": "c64"},
        # the same in double precision: the reference runs that a study checks its single-precision ones against
        {"name": "mixed_fused_c128", "kind": "circuit", "family": "mixed", "dims": "3x12,2x6", "gates": 60,
         "plan": "exhaustive", "prec": "c128"},
        # random-circuit sampling shape: layers of two-ququart Haar gates on neighbours, greedy fusion
        {"name": "brickwork_c64", "kind": "circuit", "family": "brick", "dims": "4x13", "gates": 24,
         "plan": "greedy", "prec": "c64"},
        # gate by gate from a program (no plan): one call of each kind on low, middle and high qudits
        {"name": "gate_calls_c64", "kind": "calls", "dims": "2x6,3x8,4x5", "prec": "c64"},
        # many independent small circuits of uneven size in one batch, probabilities read to the host
        {"name": "batch64", "kind": "batch", "count": 64, "gates": 200, "nmin": 6, "nmax": 11, "shape": 7},
        # the readouts that follow a circuit: norm, one marginal per kind of qudit, all probabilities
        {"name": "readout_c64", "kind": "readout", "dims": "2x8,3x4,4x7", "prec": "c64"},
        # measurement: shots drawn from the state
        {"name": "sample_c64", "kind": "sample", "dims": "3x16", "shots": 100000, "prec": "c64"},
        # the check of a single-precision run against a double-precision one
        {"name": "fidelity_c64_c128", "kind": "fidelity", "dims": "4x13", "prec": "c64"},
    ]


def _random_dims(rng, target):
    """A register of about ``target`` amplitudes: qudits of 2 to 5 levels, grouped or mixed."""
    choice = rng.choice([(2, 3), (2, 4), (3,), (2, 3, 4), (2, 3, 4, 5), (4, 3), (5, 2)])
    out, n = [], 1
    while n < target and len(out) < 28:
        d = rng.choice(choice)
        out.append(d)
        n *= d
    while len(out) > 3 and n > 1.5 * target:
        n //= out.pop(rng.randrange(len(out)))
    while len(out) < 3:
        out.append(2)
    if rng.random() < 0.5:
        out.sort(key=lambda d: choice.index(d))
    return text_of(out)


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "circuit", "circuit", "circuit", "calls", "batch", "readout", "sample", "fidelity"])
    prec = rng.choice(["c64", "c64", "c128"])
    big = 4e8 if prec == "c64" else 3e7
    if kind == "small":
        return {"kind": kind, "dims": _random_dims(rng, _log_size(rng, 16, 4000)), "gates": rng.randint(5, 120),
                "prec": "c128"}
    if kind == "circuit":
        family = rng.choice(["qutrit", "qft", "mixed", "brick"])
        plan = rng.choice(["none", "greedy", "exhaustive", "learned"])
        n = _log_size(rng, 1e3, big / (4 if plan == "none" else 1))
        if family == "qutrit":
            dims = "3x%d" % max(4, min(17, round(math.log(n, 3))))
        elif family == "qft":
            q4 = max(3, min(11, round(math.log(n, 4)) - 2))
            dims = "2x%d,4x%d" % (rng.randint(2, 6), q4)
        elif family == "brick":
            d = rng.choice([2, 3, 4, 5])
            dims = "%dx%d" % (d, max(4, round(math.log(n, d))))
        else:
            dims = _random_dims(rng, n)
        return {"kind": kind, "family": family, "dims": dims, "gates": 0 if family == "qft" else rng.randint(10, 50),
                "plan": plan, "prec": prec}
    if kind == "calls":
        return {"kind": kind, "dims": _random_dims(rng, _log_size(rng, 1e3, big)) + ",2x1,3x1", "prec": prec}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(3, 96), "gates": rng.randint(20, 200), "nmin": rng.randint(3, 6),
                "nmax": rng.randint(7, 10), "shape": rng.randrange(1 << 20)}
    dims = _random_dims(rng, _log_size(rng, 1e3, big / 2))
    if kind == "sample":
        return {"kind": kind, "dims": dims, "shots": _log_size(rng, 1, 300000), "prec": prec}
    return {"kind": kind, "dims": dims, "prec": prec}


# ------------------------------------------------------------------ gate lists
# A gate here is (kind, targets, controls, levels, param, matrix or None), the
# first listed target being the most significant local digit.

def _haar(d, rng):
    z = rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d))
    q, r = np.linalg.qr(z)
    ph = np.diag(r) / np.abs(np.diag(r))
    return np.ascontiguousarray(q * ph[None, :])


def _one(kind, dims, rng, q=None):
    n = len(dims)
    q = int(rng.integers(0, n)) if q is None else q
    if kind == "X":
        return ("X", (q,), (), None, int(rng.integers(1, dims[q])), None)
    if kind == "Z":
        return ("Z", (q,), (), None, 1, None)
    if kind == "H":
        return ("H", (q,), (), None, 0, None)
    if kind == "U1":
        return ("U", (q,), (), None, 0, _haar(dims[q], rng))
    c, t = (int(x) for x in rng.choice(n, size=2, replace=False))
    if kind == "CX":
        return ("X", (t,), (c,), (int(rng.integers(0, dims[c])),), int(rng.integers(1, dims[t])), None)
    return ("U", (c, t), (), None, 0, _haar(dims[c] * dims[t], rng))


def _circuit(case, seed):
    dims, rng = dims_of(case["dims"]), np.random.default_rng(seed)
    n, family, count = len(dims), case.get("family", "mixed"), case["gates"]
    if family == "qutrit":  # 40% Haar, 30% generalized Hadamard, 30% controlled shift
        return dims, [_one(k, dims, rng) for k in rng.choice(["U1", "H", "CX"], size=count, p=[0.4, 0.3, 0.3])]
    if family == "brick":  # neighbours (0,1), (2,3), ... then (1,2), (3,4), ...
        out, layer = [], 0
        while len(out) < count:
            for a in range(layer % 2, n - 1, 2):
                out.append(("U", (a + 1, a), (), None, 0, _haar(dims[a] * dims[a + 1], rng)))
            layer += 1
        return dims, out[:count]
    if family == "qft":
        out = [("U", (q,), (), None, 0, _haar(dims[q], rng)) for q in range(n)]
        wide = [q for q in range(n) if dims[q] == 4]
        for i in range(len(wide) - 1, -1, -1):
            out.append(("H", (wide[i],), (), None, 0, None))
            for j in range(i - 1, -1, -1):
                x = np.outer(np.arange(4), np.arange(4)).reshape(-1)
                out.append(("DIAG", (wide[j], wide[i]), (), None, 0, np.exp(2j * np.pi * x / 4.0 ** (i - j + 1))))
        bits = [q for q in range(n) if dims[q] == 2]
        for r in range(min(len(bits) - 1, len(wide))):  # Toffoli through the elevated level 2 of a ququart
            up = ("X", (wide[r],), (bits[r],), (1,), 1, None)
            out += [up, ("X", (bits[r + 1],), (wide[r],), (2,), 1, None), up[:4] + (3, None)]
        return dims, out
    return dims, [_one(k, dims, rng) for k in rng.choice(["X", "Z", "H", "CX", "U1", "U2"], size=count)]


def _calls(dims, seed):
    """One gate of each kind, on the lowest, a middle and the highest qudits."""
    rng, n = np.random.default_rng(seed), len(dims)
    lo, mid, hi = 0, n // 2, n - 1
    out = [_one("U1", dims, rng, q) for q in (lo, mid, hi)]
    out += [_one("H", dims, rng, mid), _one("X", dims, rng, hi), _one("Z", dims, rng, lo), _one("Z", dims, rng, hi)]
    out.append(("X", (mid,), (hi,), (dims[hi] - 1,), 1, None))
    out.append(("X", (lo,), (mid, hi), (0, 1), 1, None))
    x = rng.uniform(0, 2 * np.pi, dims[mid] * dims[hi])
    out.append(("DIAG", (mid, hi), (), None, 0, np.exp(1j * x)))
    out.append(("U", (mid, mid - 1), (), None, 0, _haar(dims[mid] * dims[mid - 1], rng)))
    out.append(("U", (hi,), (lo,), (1,), 0, _haar(dims[hi], rng)))
    return out


def _batch(case, seed):
    """(dims, gates) of every circuit: the sizes by the case, the gates by the seed."""
    shapes, rng = np.random.default_rng(case["shape"]), np.random.default_rng(seed)
    out = []
    for _ in range(case["count"]):
        n = int(shapes.integers(case["nmin"], case["nmax"] + 1))
        dims = [int(d) for d in shapes.choice([2, 3, 4, 5], size=n)]
        while math.prod(dims) > 1 << 20:
            dims[dims.index(max(dims))] = 2
        kinds = rng.choice(["X", "Z", "H", "CX", "U1", "U2"], size=case["gates"])
        out.append((dims, [_one(k, dims, rng) for k in kinds]))
    return out


def _records(gates):
    return [workloads.Gate(k, t, c, lv, p, m) for k, t, c, lv, p, m in gates]


def _random_state(n, prec, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    real = torch.float32 if prec == "c64" else torch.float64
    x = torch.randn(2 * n, generator=g, device="cuda", dtype=real)
    x /= torch.linalg.vector_norm(x)
    return torch.view_as_complex(x.view(n, 2))


class State:
    """What the program holds: the stream, registers on torch storage, and the handles to give back."""

    def __init__(self):
        self.stream = torch.cuda.Stream()
        self.regs, self.ends = [], []

    def register(self, dims, prec, values=None):
        n = math.prod(dims)
        buf = torch.empty(n, dtype=DTYPE[prec], device="cuda")
        torch.cuda.current_stream().synchronize()
        h = qd.qd_create(dims, None, PREC[prec], buf.data_ptr(), n * SIZE[prec], self.stream.cuda_stream)
        self.regs.append((h, buf))
        if values is not None:
            torch.cuda.synchronize()
            qd.qd_set_amplitudes(h, values.data_ptr(), qd.QD_DEVICE)
            qd.qd_sync(h)
        return h, buf

    def __del__(self):
        for end, handle in self.ends:
            end(handle)
        for h, _ in self.regs:
            qd.qd_destroy(h)


def prepare(case, seed):
    s = State()
    s.case = case
    kind = case["kind"]
    if kind == "small":
        dims, gates = _circuit(case, seed)
        s.gates = _records(gates)
        s.reg = qd.qd_create(dims, None, PREC[case["prec"]], 0, 0, s.stream.cuda_stream)
        s.regs.append((s.reg, None))
    elif kind == "circuit":
        dims, gates = _circuit(case, seed)
        s.reg, s.buf = s.register(dims, case["prec"])
        if case["plan"] == "learned":
            s.model = costmodel.load()
            qd.qd_set_cost_model(s.reg, s.model)
        s.plan = qd.qd_plan_create(s.reg, _records(gates), PLANS[case["plan"]])
        s.ends.append((qd.qd_plan_destroy, s.plan))
        if case["plan"] == "learned":
            s.ends.append((qd.qd_model_destroy, s.model))
    elif kind == "calls":
        dims = dims_of(case["dims"])
        s.reg, s.buf = s.register(dims, case["prec"], _random_state(math.prod(dims), case["prec"], seed))
        s.gates = _calls(dims, seed)
    elif kind == "batch":
        circuits = _batch(case, seed)
        s.batch = qd.qd_batch_create([d for d, _ in circuits], s.stream.cuda_stream)
        s.ends.append((qd.qd_batch_destroy, s.batch))
        for i, (_, gates) in enumerate(circuits):
            qd.qd_batch_set_circuit(s.batch, i, _records(gates))
        s.sizes = [math.prod(d) for d, _ in circuits]
        s.out = torch.empty(sum(s.sizes), dtype=torch.float64, pin_memory=True)
        host, at = s.out.numpy(), 0
        s.parts = []
        for n in s.sizes:
            s.parts.append(host[at:at + n])
            at += n
    else:
        dims = dims_of(case["dims"])
        n = math.prod(dims)
        psi = _random_state(n, case["prec"], seed)
        s.reg, s.buf = s.register(dims, case["prec"], psi)
        if kind == "readout":
            s.probs = torch.empty(n, dtype=torch.float64, device="cuda")
            s.asked = _asked(dims)
        elif kind == "sample":
            s.shots = (seed, case["shots"])
        else:
            other = psi.to(torch.complex128)
            other += 1e-3 * _random_state(n, "c128", seed + 1)
            s.other, s.obuf = s.register(dims, "c128", other)
    return s


def _asked(dims):
    """The qudits whose marginals are read: the first and the last of each dimension."""
    return sorted({dims.index(d) for d in dims} | {len(dims) - 1 - dims[::-1].index(d) for d in dims})


def run(s):
    kind = s.case["kind"]
    if kind == "small":
        qd.qd_reset(s.reg)
        qd.qd_run_circuit(s.reg, s.gates)
        idx, vals, _ = qd.qd_ket_list(s.reg)
        return [idx, vals]
    if kind == "circuit":
        qd.qd_reset(s.reg)
        qd.qd_plan_run(s.plan)
        return s.buf
    if kind == "calls":
        for k, t, c, lv, p, m in s.gates:
            if k == "U":
                qd.qd_apply(s.reg, m, t, c, lv)
            elif k == "DIAG":
                qd.qd_apply_diag(s.reg, m, t, c, lv)
            elif k == "H":
                qd.qd_apply_h(s.reg, t[0])
            elif k == "Z":
                qd.qd_apply_z(s.reg, t[0], p)
            elif not c:
                qd.qd_apply_x(s.reg, t[0], p)
            elif len(c) == 1:
                qd.qd_apply_cx(s.reg, c[0], t[0], p, lv[0])
            else:
                qd.qd_apply_mct(s.reg, c, t[0], p, lv)
        return s.buf
    if kind == "batch":
        qd.qd_batch_run(s.batch)
        for i, part in enumerate(s.parts):
            qd.qd_batch_probabilities(s.batch, i, s.sizes[i], part)
        return s.out
    if kind == "readout":
        dims = dims_of(s.case["dims"])
        norm = qd.qd_norm(s.reg)
        marginals = [qd.qd_marginal(s.reg, q, dims[q]) for q in s.asked]
        qd.qd_probabilities(s.reg, where=qd.QD_DEVICE, dev_ptr=s.probs.data_ptr())
        return [norm, np.concatenate(marginals), s.probs]
    if kind == "sample":
        return qd.qd_sample(s.reg, *s.shots)
    z = qd.qd_overlap(s.reg, s.other)
    return [z.real, z.imag, qd.qd_norm(s.other)]


# ------------------------------------------------------------------ work

def _gate_work(dims, gates):
    """(amplitudes that the gates touch, floating-point operations), summed over the gates."""
    n, amps, flops = math.prod(dims), 0.0, 0.0
    for k, t, c, lv, p, m in gates:
        share = n / math.prod(dims[q] for q in c) if c else n
        d = math.prod(dims[q] for q in t)
        if k in ("H", "U"):
            amps += share
            flops += 8.0 * d * share
        elif k in ("Z", "DIAG"):
            moved = share * (d - 1) / d if k == "Z" else share
            amps += moved
            flops += 6.0 * moved
        else:
            amps += share
    return amps, flops


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total, flops = 0, 0.0
        for dims, gates in _batch(case, 0):
            total += math.prod(dims)
            flops += _gate_work(dims, gates)[1]
        return {"bytes": 16.0 * total, "flops": flops}  # states written, probabilities written
    dims = dims_of(case["dims"])
    n, size = math.prod(dims), SIZE[case["prec"]]
    if kind == "small":
        return {"bytes": (16.0 + 24.0) * n, "flops": _gate_work(dims, _circuit(case, 0)[1])[1]}
    if kind == "circuit":
        amps, flops = _gate_work(dims, _circuit(case, 0)[1])
        # gate by gate: every touched amplitude read and written; fused: the state written by the reset,
        # then read and written once
        return {"bytes": size * n + (2.0 * size * amps if case["plan"] == "none" else 2.0 * size * n),
                "flops": flops}
    if kind == "calls":
        amps, flops = _gate_work(dims, _calls(dims, 0))
        return {"bytes": 2.0 * size * amps, "flops": flops}
    if kind == "readout":  # each of the calls reads the state
        return {"bytes": size * n * (2.0 + len(_asked(dims))) + 8.0 * n, "flops": 4.0 * n * (2 + len(_asked(dims)))}
    if kind == "sample":
        return {"bytes": size * n + 8.0 * case["shots"], "flops": 4.0 * n}
    return {"bytes": (size + 16.0 + 16.0) * n, "flops": 12.0 * n}


# ------------------------------------------------------------------ exact values

def _axes(dims, qudits):
    """The state's shape with an axis of its own for each of ``qudits``: (shape, {qudit: axis})."""
    shape, at, prev = [], {}, len(dims)
    for q in sorted(qudits, reverse=True):
        shape.append(math.prod(dims[q + 1:prev]))
        at[q] = len(shape)
        shape.append(dims[q])
        prev = q
    shape.append(math.prod(dims[:prev]))
    return shape, at


def _matrix(kind, d, power):
    w = np.exp(2j * np.pi * np.arange(d) / d)
    if kind == "H":
        return w[np.outer(np.arange(d), np.arange(d)) % d] / math.sqrt(d)
    return w[(power * np.arange(d)) % d]


def _apply(psi, dims, gate):
    kind, targets, controls, levels, param, m = gate
    shape, at = _axes(dims, list(targets) + list(controls))
    v = psi.view(shape)
    for q in sorted(controls):  # the highest axes first, so that the others keep their places
        v = v.select(at[q], levels[controls.index(q)])
        at = {p: a - (1 if a > at[q] else 0) for p, a in at.items() if p != q}
    d = [dims[q] for q in targets]
    if kind == "X":
        v.copy_(torch.roll(v, param, at[targets[0]]))
        return
    if kind in ("Z", "DIAG"):
        diag = torch.as_tensor(m if m is not None else _matrix("Z", d[0], param), device=psi.device)
        order = sorted(range(len(targets)), key=lambda i: at[targets[i]])
        diag = diag.to(torch.complex128).reshape(d).permute(order)
        new = [1] * v.dim()
        for i in order:
            new[at[targets[i]]] = d[i]
        v.mul_(diag.reshape(new))
        return
    u = torch.as_tensor(m if m is not None else _matrix("H", d[0], 0), device=psi.device).to(torch.complex128)
    front = [at[q] for q in targets]
    rest = [a for a in range(v.dim()) if a not in front]
    w = v.permute(front + rest)
    v.permute(front + rest).copy_((u @ w.reshape(u.shape[0], -1)).view(w.shape))


def _simulate(dims, gates, psi=None):
    if psi is None:
        psi = torch.zeros(math.prod(dims), dtype=torch.complex128, device="cuda")
        psi[0] = 1.0
    for g in gates:
        _apply(psi, dims, g)
    return psi


def exact(case, seed):
    kind = case["kind"]
    if kind == "sample":
        return None
    if kind == "batch":
        return torch.cat([_simulate(d, g).abs().square() for d, g in _batch(case, seed)])
    dims = dims_of(case["dims"])
    if kind in ("small", "circuit"):
        psi = _simulate(*_circuit(case, seed))
        if kind == "circuit":
            return psi
        return [None, psi[psi.abs().square() > 1e-14]]
    n = math.prod(dims)
    psi = _random_state(n, case["prec"], seed).to(torch.complex128)
    if kind == "calls":
        return _simulate(dims, _calls(dims, seed), psi)
    if kind == "readout":
        p = psi.real.square() + psi.imag.square()
        marginals = []
        for q in _asked(dims):
            shape, at = _axes(dims, [q])
            marginals.append(p.view(shape).sum((0, 2)))
        return [float(p.sum()), torch.cat(marginals), p]
    other = psi + 1e-3 * _random_state(n, "c128", seed + 1)
    z = complex(torch.vdot(psi, other))
    return [z.real, z.imag, float(other.real.square().sum() + other.imag.square().sum())]
