"""Dense matrices that fall into parts: an output's error is relative to the
members that go into it, however large the others of its group are."""
import math

import numpy as np
import pytest

from paper_2211_07918_gb300 import qudit as L
from paper_2211_07918_gb300 import workloads as wl
from test_gpu_tc_dense import DTYPE, apply_ref

pytestmark = pytest.mark.gpu
OTHERS = [7, 61, 5]  # 2,135 groups: ragged tiles of 128
PAIRS = [(2, 2), (2, 3), (3, 3), (2, 5), (3, 4), (4, 4), (3, 6), (8, 3), (3, 9), (2, 16), (4, 8)]


def matrices(a, b, rng):
    """Unitaries on (a-level, b-level) qudits with zeros between their parts."""
    d = a * b
    blocks = np.zeros((d, d), complex)
    for k in range(a):
        blocks[k * b:(k + 1) * b, k * b:(k + 1) * b] = wl.haar_unitary(b, rng)
    control = np.eye(d, dtype=complex)
    control[-b:, -b:] = blocks[:b, :b]
    return {"high alone": np.kron(wl.haar_unitary(a, rng), np.eye(b)), "low alone": np.kron(np.eye(a), blocks[:b, :b]),
            "blocks": blocks, "controlled": control,
            "moved": blocks[rng.permutation(d)][:, rng.permutation(d)]}


def members(dims, targets):
    """Of every amplitude: its group and its local index."""
    at, s = np.arange(math.prod(dims)), np.concatenate([[1], np.cumprod(dims)]).astype(int)
    loc, group = np.zeros(at.size, int), np.zeros(at.size, int)
    for q in targets:
        loc = loc * dims[q] + at // s[q] % dims[q]
    for q in range(len(dims)):
        if q not in targets:
            group = group * dims[q] + at // s[q] % dims[q]
    return group, loc


def allowed(m, psi, group, loc, prec):
    """Largest error of every output, in terms of the members that its row takes (S = sum |u| |v|, D of them,
    R and V the largest |u| and |v|).

    complex128: digits of 55 bits on the scale of V and of R, at most 2 V and 2 R: D R V 2^-55 each, and one
    rounding, below 4 D 2^-53 R V; or 2 D multiply-adds a part, each off by 2^-53 of at most S.  complex64:
    4 D multiply-adds a part (high and low words of the coefficients), each off by 2^-24 of at most S, and
    the products' own."""
    d = m.shape[0]
    v = np.zeros((group.max() + 1, d))
    v[group, loc] = np.abs(psi)
    u = np.abs(m)
    total = (v @ u.T)[group, loc]
    if prec == L.QD_C64:
        return 6 * d * 2.0 ** -24 * total + 2.0 ** -148
    couples = (u > 0).astype(float)
    top = np.stack([(v * couples[i]).max(axis=1) * u[i].max() for i in range(d)], axis=1)[group, loc]
    return 4 * d * 2.0 ** -53 * np.maximum(total, top)


def state(m, group, loc, rng, prec):
    """Random members with a magnitude of its own for each part of each group, from zero to the largest."""
    mag = [1, 1e-3, 1e-12, 1e-30, 1e-150, 0] if prec == L.QD_C128 else [1, 1e-3, 1e-9, 1e-15, 0]
    part = np.zeros(m.shape[0], int)  # of the columns: the first row that takes them
    for j in range(m.shape[0]):
        part[j] = np.flatnonzero(m[:, j])[0]
    scale = np.array(mag)[rng.integers(0, len(mag), (group.max() + 1, m.shape[0]))][group, part[loc]]
    psi = (rng.standard_normal(group.size) + 1j * rng.standard_normal(group.size)) * scale
    return psi.astype(DTYPE[prec])


def check(prec, dims, targets, m, psi, index64=0):
    group, loc = members(dims, targets)
    with L.Register(dims, None, prec) as r:
        L.qd_set_tuning(r.h, L.QD_TUNE_INDEX64, index64)
        L.qd_set_amplitudes(r.h, psi)
        L.qd_apply(r.h, m, targets)
        L.qd_sync(r.h)
        got = r.amplitudes()
    err = np.abs((got - apply_ref(psi, dims, m, targets)).astype(np.complex128))
    most = allowed(m, psi, group, loc, prec)
    assert np.all(err <= most), np.max(err / np.maximum(most, 1e-300))


@pytest.mark.parametrize("index64", [0, 1])
@pytest.mark.parametrize("kind", ["high alone", "low alone", "blocks", "controlled", "moved"])
@pytest.mark.parametrize("a,b", PAIRS)
def test_parts_have_their_own_scale(a, b, kind, index64):
    rng = np.random.default_rng(10 * a + b)
    m = matrices(a, b, rng)[kind]
    for dims, targets in (([b, a] + OTHERS, [1, 0]), ([7, b, 61, 5, a], [4, 1])):
        group, loc = members(dims, targets)
        check(L.QD_C128, dims, targets, m, state(m, group, loc, rng, L.QD_C128), index64)


@pytest.mark.parametrize("index64", [0, 1])
@pytest.mark.parametrize("dims,target", [([3, 61, 61, 17], 0), ([61, 3, 61, 17], 1), ([61, 61, 18, 3], 3)], ids=str)
def test_parts_of_three_states(dims, target, index64):
    """One state alone and two coupled, in place and moved, on registers that take the tensor cores."""
    rng = np.random.default_rng(9)
    m = np.eye(3, dtype=complex)
    m[1:, 1:] = wl.haar_unitary(2, rng)
    group, loc = members(dims, [target])
    for p, q in (([0, 1, 2], [0, 1, 2]), ([2, 0, 1], [0, 2, 1]), ([1, 2, 0], [1, 0, 2])):
        mm = m[p][:, q]
        check(L.QD_C128, dims, [target], mm, state(mm, group, loc, rng, L.QD_C128), index64)


@pytest.mark.parametrize("a,b", [(2, 5), (3, 4), (2, 7), (5, 3), (4, 4)])
@pytest.mark.parametrize("kind", ["high alone", "low alone", "blocks", "controlled", "moved"])
def test_parts_of_single_precision_gates(a, b, kind):
    rng = np.random.default_rng(10 * a + b)
    m = matrices(a, b, rng)[kind]
    for dims, targets in (([b, a] + OTHERS, [1, 0]), ([7, b, 61, 5, a], [4, 1])):
        group, loc = members(dims, targets)
        check(L.QD_C64, dims, targets, m, state(m, group, loc, rng, L.QD_C64))


@pytest.mark.parametrize("prec", [L.QD_C64, L.QD_C128])
@pytest.mark.parametrize("d", [4, 9, 16, 27])
def test_rows_that_share_members_or_hold_small_entries(d, prec):
    """Rows that overlap without being alike, and entries of very different size: sums of rounded products."""
    rng = np.random.default_rng(d)
    ring = np.zeros((d, d), complex)
    for i in range(d):
        ring[i, [i, (i + 1) % d]] = rng.standard_normal(2) + 1j * rng.standard_normal(2)
    small = wl.haar_unitary(d, rng)
    small[:, 1] *= 1e-9
    dims = [d] + OTHERS
    group, loc = members(dims, [0])
    for m, largest in ((ring, 0), (small, 1)):
        psi = rng.standard_normal(group.size) + 1j * rng.standard_normal(group.size)
        psi[loc != largest] *= 1e-9
        check(prec, dims, [0], m, psi.astype(DTYPE[prec]))


@pytest.mark.parametrize("dims,targets,run", [
    ([2] * 15, [3, 0], [(4, 6), (9,)]), ([3, 3, 7, 4, 61], [1, 0], [(2, 3), (0,)]), ([4, 3, 7, 4, 61], [0, 1], [(2, 3)]),
    ([4, 7, 4, 4, 61], [2, 0], [(1, 3), (2,)])], ids=str)
def test_parts_with_a_run(dims, targets, run):
    rng = np.random.default_rng(6)
    a, b = dims[targets[0]], dims[targets[1]]
    group, loc = members(dims, targets)
    s = np.concatenate([[1], np.cumprod(dims)]).astype(int)
    for m in matrices(a, b, rng).values():
        psi = state(m, group, loc, rng, L.QD_C128)
        gates, want = [wl.Gate("U", tuple(targets), matrix=m)], apply_ref(psi, dims, m, targets)
        for qs in run:
            phases = np.exp(2j * np.pi * rng.random(math.prod(dims[q] for q in qs)))
            gates.append(wl.Gate("DIAG", tuple(qs), matrix=phases))
            at = np.zeros(group.size, int)
            for q in qs:
                at = at * dims[q] + np.arange(group.size) // s[q] % dims[q]
            want = want * phases[at].astype(np.clongdouble)
        with L.Register(dims, None, L.QD_C128) as r:
            L.qd_set_amplitudes(r.h, psi)
            plan = L.qd_plan_create_forms(r.h, gates, [(0, len(gates) - 1)], [L.QD_FORM_DENSE_RUN])
            L.qd_plan_run(plan)
            L.qd_sync(r.h)
            got = r.amplitudes()
            L.qd_plan_destroy(plan)
        # the table's entry took one complex product per gate of the run, and one more multiplies the output
        most = allowed(m, psi, group, loc, L.QD_C128) + 4 * (len(run) + 1) * 2.0 ** -53 * np.abs(want.astype(complex))
        assert np.all(np.abs((got - want).astype(np.complex128)) <= most)


@pytest.mark.parametrize("a,b", [(2, 2), (3, 3), (2, 16)])
def test_special_values_in_one_part(a, b):
    """A part that holds an infinity or only extremely small numbers takes its whole group to FP64, as every
    member times a zero entry does there; other groups are not affected."""
    rng = np.random.default_rng(1)
    m = matrices(a, b, rng)["blocks"]
    dims, targets = [b, a] + OTHERS, [1, 0]
    group, loc = members(dims, targets)
    psi = rng.standard_normal(group.size) + 1j * rng.standard_normal(group.size)
    psi[(group % 11 == 3) & (loc == 0)] = np.inf
    psi[(group % 11 == 5) & (loc < b)] *= 1e-290
    psi[(group % 11 == 7) & (loc < b)] *= 1e-321  # denormal numbers
    fine = group % 11 != 3
    with L.Register(dims, None, L.QD_C128) as r:
        L.qd_set_amplitudes(r.h, psi)
        L.qd_apply(r.h, m, targets)
        L.qd_sync(r.h)
        got = r.amplitudes()
    with np.errstate(all="ignore"):
        want = apply_ref(psi, dims, m, targets)
    most = allowed(m, np.where(fine, psi, 0), group, loc, L.QD_C128) + 2 * a * b * 2.0 ** -1074
    assert np.all(np.abs((got[fine] - want[fine]).astype(np.complex128)) <= most[fine])
    assert not np.any(np.isfinite(got.real[~fine]) & np.isfinite(got.imag[~fine]))


@pytest.mark.parametrize("d,dims", [(2, [2, 5, 61, 61, 17]), (3, [3, 61, 61, 17]), (4, [4] + OTHERS), (9, [9] + OTHERS), (27, [27] + OTHERS)])
def test_groups_of_denormal_numbers(d, dims):
    rng = np.random.default_rng(d)
    psi = (rng.integers(-2000, 2000, math.prod(dims)) + 1j * rng.integers(-2000, 2000, math.prod(dims))) * 2.0 ** -1074
    m = wl.haar_unitary(d, rng)
    with L.Register(dims, None, L.QD_C128) as r:
        L.qd_set_amplitudes(r.h, psi)
        L.qd_apply(r.h, m, [0])
        L.qd_sync(r.h)
        got = r.amplitudes()
    # every product is rounded to a multiple of 2^-1074: 2 D multiply-adds a part, half a unit each
    err = np.abs((got - apply_ref(psi, dims, m, [0])).astype(np.clongdouble))
    assert np.max(err) <= 2 * d * np.longdouble(2) ** -1074


def test_norm_after_many_gates_of_16_states():
    """200 single-precision gates of 16 states: the norm drifts by no more than the roundings of the outputs.

    A part is off by 2^-26 of its group's largest and rounded to 2^-24 of itself four times, without a
    preferred sign: over the 1.3e5 parts a gate moves the norm by 2 0.5 2^-24 sqrt(3 / 1.3e5) = 3e-10 (one
    deviation), 200 gates by 4e-9, four deviations 1.7e-8.  The matrix is held to 2^-36: below
    2^-36 sqrt(16) a gate, 1.2e-8 for 200 of one sign."""
    rng = np.random.default_rng(3)
    dims = [4] * 8
    psi = rng.standard_normal(4 ** 8) + 1j * rng.standard_normal(4 ** 8)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64)
    gates = []
    for i in range(200):
        q = int(rng.integers(0, 7))
        gates.append(wl.Gate("U", (q, q + 1), matrix=wl.haar_unitary(16, rng)))
    with L.Register(dims, None, L.QD_C64) as r:
        L.qd_set_amplitudes(r.h, psi)
        before = L.qd_norm(r.h)
        r.run(gates, L.QD_PLAN_NONE)
        after = L.qd_norm(r.h)
    assert abs(after - before) <= 3e-8


def unusual(kind, d, rng, prec):
    """Matrices outside the exponents that the digits of qd_tc32.cu and qd_tc64.cu hold."""
    m = wl.haar_unitary(d, rng)
    far = 30 if prec == L.QD_C64 else 150
    if kind == "small":
        return m * 2.0 ** -far
    if kind == "large":
        return m * 2.0 ** far
    m[1] *= 2.0 ** (-12 if prec == L.QD_C64 else -far)
    return m


@pytest.mark.parametrize("kind", ["small", "large", "one row"])
@pytest.mark.parametrize("dims", [[3, 3], [4, 3], [2, 7], [4, 4]], ids=str)
def test_blocks_of_unusual_matrices(dims, kind):
    """Tensor-core blocks of 9 to 16 states that run on the kernel of the larger ones: parts in three BF16
    slices, 2^-27 of a scale of at most 2 V (the group's largest), rows likewise of 2 R, and three
    roundings of at most D R V: below D 2^-22 R V for every row."""
    rng = np.random.default_rng(2)
    d = math.prod(dims)
    regs, targets = dims + OTHERS, [1, 0]
    first = wl.haar_unitary(d, rng)
    m = unusual(kind, d, rng, L.QD_C64)
    gates = [wl.Gate("U", tuple(targets), matrix=first), wl.Gate("U", tuple(targets), matrix=m @ first.conj().T)]
    group, loc = members(regs, targets)
    psi = (rng.standard_normal(group.size) + 1j * rng.standard_normal(group.size)).astype(np.complex64)
    for index64 in (0, 1):
        with L.Register(regs, None, L.QD_C64) as r:
            L.qd_set_tuning(r.h, L.QD_TUNE_INDEX64, index64)
            L.qd_set_amplitudes(r.h, psi)
            plan = L.qd_plan_create_forms(r.h, gates, [(0, 1)], [L.QD_FORM_BLOCK_TC])
            L.qd_plan_run(plan)
            L.qd_sync(r.h)
            got = r.amplitudes()
            L.qd_plan_destroy(plan)
        err = np.abs((got - apply_ref(psi, regs, m, targets)).astype(complex))
        v = np.zeros(group.max() + 1)
        np.maximum.at(v, group, np.abs(psi))
        assert np.all(err <= d * 2.0 ** -22 * v[group] * np.abs(m).max(axis=1)[loc])


@pytest.mark.parametrize("prec", [L.QD_C64, L.QD_C128])
@pytest.mark.parametrize("kind", ["small", "large", "one row"])
@pytest.mark.parametrize("d", [4, 9, 12, 16, 27])
def test_gates_of_unusual_matrices(d, kind, prec):
    rng = np.random.default_rng(d)
    m = unusual(kind, d, rng, prec)
    dims = [7, d, 61, 5]
    group, loc = members(dims, [1])
    psi = (rng.standard_normal(group.size) + 1j * rng.standard_normal(group.size)).astype(DTYPE[prec])
    check(prec, dims, [1], m, psi)
    if prec == L.QD_C128 and d <= 16:  # with a run: the table of a phase per level of qudit 0
        phases = np.exp(2j * np.pi * rng.random(7))
        gates = [wl.Gate("U", (1,), matrix=m), wl.Gate("DIAG", (0,), matrix=phases)]
        with L.Register(dims, None, prec) as r:
            L.qd_set_amplitudes(r.h, psi)
            plan = L.qd_plan_create_forms(r.h, gates, [(0, 1)], [L.QD_FORM_DENSE_RUN])
            L.qd_plan_run(plan)
            L.qd_sync(r.h)
            got = r.amplitudes()
            L.qd_plan_destroy(plan)
        want = apply_ref(psi, dims, m, [1]) * phases[np.arange(group.size) % 7]
        most = allowed(m, psi, group, loc, prec) + 4 * 2.0 ** -53 * np.abs(want.astype(complex))
        assert np.all(np.abs((got - want).astype(np.complex128)) <= most)
