"""Readouts whose sums run on the integer units, at the edges of their tiles
and value ranges, against 64-bit numpy."""
import math

import numpy as np
import pytest

from paper_2211_07918_gb300 import qudit as L

pytestmark = pytest.mark.gpu

DTYPE = {L.QD_C64: np.complex64, L.QD_C128: np.complex128}
# below, at and above the blocks' tiles; odd sizes; qudits of short period, of longer period, of many levels
SHAPES = [[2, 2, 2], [3, 5, 7], [2] * 12, [3] * 8, [64, 5, 3], [3, 64, 64], [2] * 8 + [3] * 4, [3] * 11 + [2, 2, 3], [8, 256 // 8, 9, 7], [3] * 13]


def state(n, prec, seed, kind):
    rng = np.random.default_rng(seed)
    z = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    if kind == "wide":  # parts over the whole range of the type's squares
        z = z * 10.0 ** rng.uniform(-30 if prec == L.QD_C64 else -120, 2, n)
        z.imag *= 10.0 ** rng.uniform(-20, 0, n)
    elif kind == "sparse":
        z[rng.random(n) < 0.97] = 0
        z[-1] = 0.5
    else:
        z /= np.linalg.norm(z)
    return z.astype(DTYPE[prec])


def probs(z):
    x, y = z.real.astype(np.float64), z.imag.astype(np.float64)
    return x * x + y * y


@pytest.mark.parametrize("prec", [L.QD_C64, L.QD_C128])
@pytest.mark.parametrize("kind", ["unit", "wide", "sparse"])
@pytest.mark.parametrize("dims", SHAPES, ids=str)
def test_norm_marginals_probabilities_overlap(dims, kind, prec):
    n = math.prod(dims)
    z, w = state(n, prec, 1, kind), state(n, L.QD_C128, 2, kind)
    p = probs(z)
    with L.Register(dims, None, prec) as r, L.Register(dims, None, L.QD_C128) as q, L.Register(dims, None, prec) as t:
        L.qd_set_amplitudes(r.h, z)
        L.qd_set_amplitudes(q.h, w)
        L.qd_set_amplitudes(t.h, w.astype(DTYPE[prec]))
        # a group is truncated by at most 16 units of 2^-57 of its largest square; a thread and the
        # block trees add at most some 40 terms in FP64 here: 40 2^-53 < 1e-14 of the sum
        assert abs(L.qd_norm(r.h) - math.fsum(p)) <= 1e-14 * math.fsum(p)
        shaped = p.reshape(dims[::-1])
        for k, d in enumerate(dims):
            got = L.qd_marginal(r.h, k, d)
            want = [math.fsum(np.take(shaped, x, axis=len(dims) - 1 - k).ravel()) for x in range(d)]
            assert np.all(np.abs(got - want) <= 1e-14 * np.array(want))
        got = L.qd_probabilities(r.h)
        if prec == L.QD_C64:
            assert np.array_equal(got, p)  # exact squares, one rounding
        else:
            assert np.all(np.abs(got - p) <= 2.0 ** -52 * p)
        for other, b in ((q, w), (t, w.astype(DTYPE[prec]))):
            a, c = z.astype(np.complex128), b.astype(np.complex128)
            scale = math.fsum(np.abs(a) * np.abs(c))
            prod = [a.real * c.real, a.imag * c.imag, a.real * c.imag, -a.imag * c.real]
            got = L.qd_overlap(r.h, other.h)
            # products truncated to 2^-57 of the group's largest |a||b|, sums as above; the products
            # of the reference are rounded (2^-53 of each)
            assert abs(got.real - math.fsum(np.concatenate(prod[:2]))) <= 2e-14 * scale
            assert abs(got.imag - math.fsum(np.concatenate(prod[2:]))) <= 2e-14 * scale


def test_probabilities_of_special_values():
    tiny, inf, nan = np.float32(1e-45), np.inf, np.nan
    parts = [0.0, -0.0, tiny, -3 * tiny, np.float32(1.1754944e-38), 1.5, -2.0 ** -60, 3e38, inf, -inf, nan, 1 + 2.0 ** -23]
    z = np.array([complex(np.float32(a), np.float32(b)) for a in parts for b in parts], dtype=np.complex64)
    with L.Register([12, 12], None, L.QD_C64) as r:
        L.qd_set_amplitudes(r.h, z)
        got = L.qd_probabilities(r.h)
        assert np.array_equal(got, probs(z), equal_nan=True)
        assert math.isnan(L.qd_norm(r.h))
        z[~np.isfinite(z)] = 0
        L.qd_set_amplitudes(r.h, z)
        assert abs(L.qd_norm(r.h) - math.fsum(probs(z))) <= 1e-14 * math.fsum(probs(z))
        z[np.abs(z) > 1e-30] = 0  # only denormals and smallest normals are left
        L.qd_set_amplitudes(r.h, z)
        assert abs(L.qd_norm(r.h) - math.fsum(probs(z))) <= 1e-14 * math.fsum(probs(z)) and L.qd_norm(r.h) > 0


@pytest.mark.parametrize("prec", [L.QD_C64, L.QD_C128])
@pytest.mark.parametrize("kind", ["unit", "sparse"])
@pytest.mark.parametrize("dims", [[2, 2, 2], [3, 5, 7], [2] * 12, [17, 61, 4], [3] * 14], ids=str)
def test_sampling_levels(dims, kind, prec):
    n = math.prod(dims)
    z = state(n, prec, 3, kind)
    if n > 50000:
        z[4096 * 100:4096 * 1030] = 0  # empty chunks across two supers
    p = probs(z)
    cdf = np.cumsum(p.astype(np.longdouble))
    rng = np.random.default_rng(4)
    u = np.concatenate([rng.random(3000), [0.0, 1 - 2.0 ** -53, 1.0, 2.0, -0.5, np.nan]])
    with L.Register(dims, None, prec) as r:
        L.qd_set_amplitudes(r.h, z)
        got = L.qd_sample_u(r.h, u)
        assert np.array_equal(L.qd_sample(r.h, 9, 1000)[:10], L.qd_sample(r.h, 9, 10))  # a shot's draw is its own
    assert got[-1] == got[-3] == got[-4] == n - 1 and got[-2] == 0
    g, t = got[:-4], u[:-4] * float(cdf[-1])
    # the target lies in the drawn amplitude's interval up to the rounding of the prefix sums
    eps = 1e-13 * float(cdf[-1])
    assert np.all(p[g] > 0)
    assert np.all(cdf[g] >= t - eps) and np.all(cdf[g] - p[g] <= t + eps)
