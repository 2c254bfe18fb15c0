"""Circuits on a stream of their own, where kernels of small and middle-sized registers are launched before
the ones they follow have ended: the same states, to the bit, as on the default stream, which orders whole
kernels."""
import math

import numpy as np
import pytest
import torch

from paper_2211_07918_gb300 import qudit as L
from paper_2211_07918_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def circuit(dims, count, seed):
    """Gates of every kind on all qudits; dense ones of one and two qudits, some in parts, runs of diagonals."""
    rng, n, out = np.random.default_rng(seed), len(dims), []
    while len(out) < count:
        q, p = (int(x) for x in rng.choice(n, 2, replace=False))
        d = dims[q] * dims[p]
        kind = rng.integers(0, 8)
        if kind == 0:
            out.append(wl.Gate("X", (q,), param=1))
        elif kind == 1:
            out.append(wl.Gate("Z", (q,), param=1))
        elif kind == 2:
            out.append(wl.Gate("X", (q,), (p,), (0,), 1))
        elif kind == 3:
            out.append(wl.Gate("H", (q,)))
        elif kind == 4:
            out.append(wl.Gate("U", (q,), matrix=wl.haar_unitary(dims[q], rng)))
        elif kind == 5 and d <= 32:
            out.append(wl.Gate("U", (q, p), matrix=wl.haar_unitary(d, rng)))
        elif kind == 6 and d <= 32:
            out.append(wl.Gate("U", (q, p), matrix=np.kron(wl.haar_unitary(dims[q], rng), np.eye(dims[p]))))
        elif kind == 7 and d <= 32:
            out += [wl.Gate("H", (q,)), wl.Gate("DIAG", (q, p), matrix=np.exp(2j * np.pi * rng.random(d)))]
    return out


def run(dims, gates, prec, how, stream, repeats):
    """The state after `repeats` passes, with a readout behind the last one, and the norm."""
    with L.Register(dims, None, prec, stream=stream) as r:
        if how == "calls":
            for _ in range(repeats):
                L.qd_reset(r.h)
                for g in gates:
                    L.qd_apply_gate(r.h, g)
        else:
            plan = L.qd_plan_create(r.h, gates, how)
            for _ in range(repeats):  # on a stream of its own the first pass is captured, the later ones replayed
                L.qd_reset(r.h)
                L.qd_plan_run(plan)
        norm = L.qd_norm(r.h)
        assert L.qd_sync(r.h) == 0
        state = r.amplitudes()
        if how != "calls":
            L.qd_plan_destroy(plan)
    return state, norm


@pytest.mark.parametrize("prec", [L.QD_C64, L.QD_C128])
@pytest.mark.parametrize("how", ["calls", L.QD_PLAN_NONE, L.QD_PLAN_GREEDY, L.QD_PLAN_EXHAUSTIVE])
@pytest.mark.parametrize("dims", [[2] * 10, [3] * 6 + [2], [4, 3, 2, 5, 4, 3], [2] * 14, [4] * 8, [3] * 11, [2] * 17, [5, 3, 4, 2, 3, 5, 4, 3, 2, 4],
                                  [3] * 13, [4] * 10 + [2], [8, 16, 4, 9, 27, 2]], ids=str)
def test_chained_launches_leave_the_same_state(dims, how, prec):
    gates = circuit(dims, 60, len(dims))
    stream = torch.cuda.Stream()
    want, norm = run(dims, gates, prec, how, 0, 1)
    for repeats in (1, 3):
        got, n = run(dims, gates, prec, how, stream.cuda_stream, repeats)
        assert np.array_equal(got, want) and n == norm


@pytest.mark.parametrize("prec", [L.QD_C64, L.QD_C128])
@pytest.mark.parametrize("d,n", [(2, 1 << 10), (2, 1 << 15), (2, 1 << 20), (2, 1 << 22), (3, 3 ** 7), (3, 3 ** 10), (3, 3 ** 12), (3, 3 ** 14),
                                 (4, 1 << 10), (4, 1 << 16), (4, 1 << 20), (8, 1 << 12), (8, 1 << 18), (8, 1 << 21), (16, 1 << 12),
                                 (16, 1 << 20), (9, 3 ** 10), (27, 3 ** 9), (27, 3 ** 13), (32, 1 << 15), (32, 1 << 20)])
def test_one_kernel_after_itself(d, n, prec):
    """Sixty gates of one dimension, dense, in parts, permuting and diagonal, in turn and alone."""
    rng = np.random.default_rng(d)
    base = next(b for b in (2, 3) if round(b ** round(math.log(d, b))) == d)
    k, count = round(math.log(d, base)), round(math.log(n, base))
    dims = [base] * count
    kinds = {"dense": [], "parts": [], "permuting": [], "diagonal": []}
    for i in range(60):
        t = tuple((i * 5 + 1 + j) % count for j in range(k))
        m = wl.haar_unitary(d, rng)
        perm = np.eye(d)[rng.permutation(d)] * np.exp(2j * np.pi * rng.random(d))
        kinds["dense"].append(wl.Gate("U", t, matrix=m))
        kinds["parts"].append(wl.Gate("U", t, matrix=np.kron(np.eye(base), wl.haar_unitary(d // base, rng)) if k > 1 else m))
        kinds["permuting"].append(wl.Gate("U", t, matrix=perm))
        kinds["diagonal"].append(wl.Gate("DIAG", t, matrix=np.exp(2j * np.pi * rng.random(d))))
    kinds["in turn"] = [kinds[x][i] for i in range(15) for x in ("dense", "diagonal", "parts", "permuting")]
    stream = torch.cuda.Stream()
    for gates in kinds.values():
        want, norm = run(dims, gates, prec, L.QD_PLAN_NONE, 0, 1)
        got, other = run(dims, gates, prec, L.QD_PLAN_NONE, stream.cuda_stream, 2)
        assert np.array_equal(got, want) and norm == other
