"""Dense gates on the tensor cores in both precisions: every dimension, slot
layout, ragged tiles, controls and both index widths against extended precision."""
import math

import numpy as np
import pytest

from paper_2211_07918_gb300 import qudit as L
from paper_2211_07918_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
BOTH = [L.QD_C64, L.QD_C128]
DTYPE = {L.QD_C64: np.complex64, L.QD_C128: np.complex128}


def bound(prec, d):
    """Largest error of a part of the result of a unitary gate, in units of the group's largest part.

    complex128: 2 D products of parts off by at most half a last place of the largest, the matrix
    entries likewise, one rounding of the result: below 4 D 2^-53.  complex64: parts off by 2^-26 of
    the largest, sqrt(2 D) in sum, and four FP32 roundings of a result of at most sqrt(2 D):
    below sqrt(2 D) 2^-22."""
    return 4 * d * 2.0 ** -53 if prec == L.QD_C128 else math.sqrt(2 * d) * 2.0 ** -22


def apply_ref(psi, dims, m, targets, controls=(), levels=()):
    """psi after the gate, in extended precision."""
    n = len(dims)
    t = psi.astype(np.clongdouble).reshape(dims[::-1]).copy()
    view = t[tuple(levels[controls.index(q)] if q in controls else slice(None) for q in range(n - 1, -1, -1))]
    left = [q for q in range(n - 1, -1, -1) if q not in controls]
    front = [left.index(q) for q in targets]
    w = np.moveaxis(view, front, range(len(front)))
    d = m.shape[0]
    out = np.matmul(m.astype(np.clongdouble), w.reshape(d, -1)).reshape(w.shape)
    w[...] = out
    return t.ravel()


def check(prec, dims, targets, controls=(), levels=(), index64=0, seed=0, scale=1.0, limit=None):
    rng = np.random.default_rng(seed)
    n, d = math.prod(dims), math.prod(dims[q] for q in targets)
    psi = (rng.standard_normal(n) + 1j * rng.standard_normal(n)) * scale
    psi[rng.random(n) < 0.05] = 0
    psi = psi.astype(DTYPE[prec])
    m = wl.haar_unitary(d, rng)
    with L.Register(dims, None, prec) as r:
        L.qd_set_tuning(r.h, L.QD_TUNE_INDEX64, index64)
        L.qd_set_amplitudes(r.h, psi)
        L.qd_apply(r.h, m, targets, controls, levels or None)
        L.qd_sync(r.h)
        got = r.amplitudes()
    want = apply_ref(psi, dims, m, targets, tuple(controls), tuple(levels))
    err = np.max(np.abs((got - want).astype(np.complex128)))
    assert err <= (limit or bound(prec, d)) * np.max(np.abs(psi)), (err, d)
    if controls:  # amplitudes outside the control slice are untouched
        same = apply_ref(psi, dims, np.zeros((d, d)), targets, tuple(controls), tuple(levels)) != 0
        assert np.array_equal(got[same], psi[same])


@pytest.mark.parametrize("prec", BOTH)
@pytest.mark.parametrize("index64", [0, 1])
@pytest.mark.parametrize("d", list(range(2, 33)))
def test_every_dimension(d, index64, prec):
    # 1 qudit of d levels below, inside and above others; a group count that fills no tile evenly
    n_other = {2: 310000, 3: 190000}.get(d, 17000) // d // 7 + 1
    a = next(x for x in range(64, 1, -1) if n_other / x > 1)
    b = min(64, n_other // a + 1)
    c = max(2, -(-n_other // (a * b)))
    for dims, t in (([d, 7, a, b, c], 0), ([7, a, d, b, c], 2), ([7, c, a, b, d], 4)):
        assert math.prod(dims) >= {2: 300000, 3: 180000}.get(d, 16384)
        check(prec, dims, [t], index64=index64, seed=d)


@pytest.mark.parametrize("d", [10, 13, 16])
@pytest.mark.parametrize("others", [(64, 32, 19), (64, 61, 10), (64, 64, 19), (64, 47, 26), (64, 63, 29), (64, 61, 30)])
def test_sizes_around_the_cuda_core_wave(d, others):
    """Groups from 256 to 768 for each of 152 SMs, where single complex64 gates change kernels.  The
    CUDA cores add 2 D products in FP32, each sum below sqrt(2 D): at most 2 D sqrt(2 D) 2^-24."""
    check(L.QD_C64, [others[0], d, *others[1:]], [1], seed=d, limit=2 * d * math.sqrt(2 * d) * 2.0 ** -24)


@pytest.mark.parametrize("prec", BOTH)
@pytest.mark.parametrize("dims,targets,controls,levels", [
    ([2] * 17, [3, 9], [], []), ([2] * 17, [0, 1, 2], [], []), ([2] * 18, [16, 2, 7, 5], [4], [0]),
    ([3] * 11, [4, 0], [], []), ([3] * 11, [0, 1, 2], [], []), ([3] * 14, [7], [0, 3], [2, 1]),
    ([4, 3, 2] * 4, [0, 3], [1], [1]), ([5, 2, 4, 3, 4, 5, 3, 4, 4], [5, 0], [], []),
    ([2, 64, 9, 16], [0, 3], [], []), ([3] * 12 + [2, 2], [13], [12], [1])], ids=str)
def test_geometries(dims, targets, controls, levels, prec):
    check(prec, dims, targets, controls, levels, seed=3)
    check(prec, dims, targets, controls, levels, seed=4, scale=1e-90 if prec == L.QD_C128 else 1e-15)


@pytest.mark.parametrize("prec", BOTH)
@pytest.mark.parametrize("dims,target", [([2] * 19, 4), ([3] * 11 + [2], 2), ([5] * 7, 1), ([20, 4, 5, 5, 9], 0), ([31, 9, 8, 8], 0)],
                         ids=str)
def test_groups_outside_the_integers_range(dims, target, prec):
    """Infinities, NaN, and groups of extremely small or large amplitudes go through FP64; their
    neighbours are not affected, and a group keeps its own scale."""
    rng = np.random.default_rng(5)
    n, d = math.prod(dims), dims[target]
    psi = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    s = math.prod(dims[:target])
    group = np.arange(n) // (s * d) * s + np.arange(n) % s
    kind = group % 97
    psi[kind == 1] *= 1e-250 if prec == L.QD_C128 else 1e-34
    psi[kind == 2] *= 1e+290 if prec == L.QD_C128 else 1e+34
    psi[kind == 3] *= 1e-12
    psi[kind == 4] = 0
    psi[(kind == 5) & (np.arange(n) // s % d == 1)] = np.inf
    psi[(kind == 6) & (np.arange(n) // s % d == 0)] = complex(np.nan, 1)
    psi = psi.astype(DTYPE[prec])
    m = wl.haar_unitary(d, rng)
    with L.Register(dims, None, prec) as r:
        L.qd_set_amplitudes(r.h, psi)
        L.qd_apply(r.h, m, [target])
        L.qd_sync(r.h)
        got = r.amplitudes()
    with np.errstate(all="ignore"):
        want = apply_ref(psi, dims, m, [target])
    fine = (kind != 5) & (kind != 6)
    largest = np.zeros(group.max() + 1)
    np.maximum.at(largest, group[fine], np.abs(psi[fine]))
    floor = 0 if prec == L.QD_C128 else 2.0 ** -148  # results below the normal numbers
    assert np.all(np.abs((got[fine] - want[fine]).astype(np.complex128)) <= bound(prec, d) * largest[group[fine]] + floor)
    assert not np.any(np.isfinite(got.real[~fine]) & np.isfinite(got.imag[~fine]))


@pytest.mark.parametrize("prec", BOTH)
@pytest.mark.parametrize("d", [2, 3, 4, 7, 9, 16, 20, 27, 32])
def test_leading_digits_at_their_limits(d, prec):
    """Amplitudes and matrix entries just below, at and above powers of two."""
    rng = np.random.default_rng(d)
    n_other = {2: 300000, 3: 180000}.get(d, 20000) // d // 8 + 1
    dims = [4, d, 2, 64, min(64, n_other // 64 + 2), n_other // 4096 + 2]
    near = np.array([s * (1 + t * 2.0 ** -k) for s in (1, -1) for t in (1, -1, 0) for k in range(1, 54)])
    n = math.prod(dims)
    psi = (rng.choice(near, n) + 1j * rng.choice(near, n)).astype(DTYPE[prec])
    m = rng.choice(near, (d, d)) + 1j * rng.choice(near, (d, d))
    with L.Register(dims, None, prec) as r:
        L.qd_set_amplitudes(r.h, psi)
        L.qd_apply(r.h, m, [1])
        L.qd_sync(r.h)
        got = r.amplitudes()
    # matrix rows of largest part up to 1.5, amplitudes up to 1.5, 2 D products of parts, each side
    # off by half a last place of the largest: 2 D (2 2^-53 1.5 1.5) and one rounding; complex64:
    # 2 D 2.25 (2^-26 and four roundings of 2^-24)
    err = np.max(np.abs((got - apply_ref(psi, dims, m, [1])).astype(np.complex128)))
    assert err <= (12 * d * 2.0 ** -53 if prec == L.QD_C128 else 6 * d * 2.0 ** -23), err


@pytest.mark.parametrize("index64", [0, 1])
@pytest.mark.parametrize("dims,targets,run", [
    ([2] * 19, [4], [(3, 6), (9,), (2, 5)]), ([3] * 11 + [2], [0], [(1, 4), (0,)]), ([4] * 8, [5], [(0, 2), (7,)]),
    ([5, 3, 7, 2, 4, 5, 6], [2], [(0, 3), (5,)]), ([3] * 10, [8, 1], [(2, 5), (9, 0)]), ([2, 3, 4, 5, 6, 7, 5], [1, 3], [(2, 6)]),
    ([4] * 8, [0, 3], [(1, 6), (2,)]), ([2] * 15, [3, 0, 8, 9], [(12, 3), (1,)])], ids=str)
def test_dense_part_with_a_run(dims, targets, run, index64):
    """A dense part followed by a diagonal run in one launch, against the oracle of its gates."""
    rng = np.random.default_rng(2)
    n, d = math.prod(dims), math.prod(dims[q] for q in targets)
    m = wl.haar_unitary(d, rng)
    psi = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    s = np.concatenate([[1], np.cumprod(dims)]).astype(int)
    gates = [wl.Gate("U", tuple(targets), matrix=m)]
    want = apply_ref(psi, dims, m, targets)
    for qs in run:
        phases = np.exp(2j * np.pi * rng.random(math.prod(dims[q] for q in qs)))
        gates.append(wl.Gate("DIAG", tuple(qs), matrix=phases))
        loc = np.zeros(n, int)
        for q in qs:
            loc = loc * dims[q] + np.arange(n) // s[q] % dims[q]
        want = want * phases[loc].astype(np.clongdouble)
    with L.Register(dims, None, L.QD_C128) as r:
        L.qd_set_tuning(r.h, L.QD_TUNE_INDEX64, index64)
        L.qd_set_amplitudes(r.h, psi)
        plan = L.qd_plan_create_forms(r.h, gates, [(0, len(gates) - 1)], [L.QD_FORM_DENSE_RUN])
        L.qd_plan_run(plan)
        L.qd_sync(r.h)
        got = r.amplitudes()
        L.qd_plan_destroy(plan)
    # the gate as above, then one complex product (two roundings a part) with a table of phases that
    # took one complex product per gate of the run
    top = np.max(np.abs(psi))
    assert np.max(np.abs((got - want).astype(np.complex128))) <= (4 * d + 4 * math.sqrt(d) * (len(run) + 1)) * 2.0 ** -53 * top


def test_fused_plan_matches_single_gates():
    dims = [3, 2, 4, 3, 2, 3, 4, 3, 2, 3, 2]
    gates = wl.random_circuit(dims, 60, 11, wl.C0_MIX + ("U2",))
    out = []
    for kind in (L.QD_PLAN_NONE, L.QD_PLAN_GREEDY, L.QD_PLAN_EXHAUSTIVE):
        with L.Register(dims, None, L.QD_C128) as r:
            r.run(gates, kind)
            L.qd_sync(r.h)
            out.append(r.amplitudes())
    for o in out[1:]:
        assert np.max(np.abs(o - out[0])) <= 1e-13
