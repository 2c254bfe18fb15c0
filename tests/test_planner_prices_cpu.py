"""Prices of the planner's analytic model against measured launches (host only)."""
import numpy as np
import pytest

from paper_2211_07918_gb300 import qudit as L
from paper_2211_07918_gb300 import workloads as wl
from paper_2211_07918_gb300.build import build
from paper_2211_07918_gb300.workloads import Gate

N17 = 3 ** 17


@pytest.fixture(scope="module", autouse=True)
def _built():
    build()


def dense(qudits, d, seed=0):
    return Gate("U", tuple(qudits), matrix=wl.haar_unitary(d, np.random.default_rng(seed)))


def cost(gates, dims=(3,) * 17, prec=L.QD_C64):
    return L.qd_debug_segment_cost(list(dims), gates, 0, len(gates) - 1, prec)


def test_wide_blocks_are_not_priced_below_their_slowest_place():
    """A three-qutrit block on qudits 0 to 2 of 17 moves 2.79 TB/s: 741 us."""
    assert cost([dense((0, 1), 9), dense((1, 2), 9)]) >= 0.9 * 2 * 8 * N17 / 2.79e12


def test_complex128_matrices_that_stay_on_the_fp64_pipe():
    """The product of a gate, a controlled shift on its qudit's neighbour and another gate has rows that share
    some of their members: 4 D multiply-adds an amplitude; without the first gate it falls into parts."""
    shift, first, last = Gate("X", (4,), (5,), (1,), 1), dense((5,), 3, 1), dense((5,), 3, 2)
    _, m = L.qd_debug_fuse_block([3] * 17, [first, shift, last], 0, 2)
    rows = m != 0
    assert any(0 < np.sum(a & b) < np.sum(a) for a in rows for b in rows)
    on_pipe = N17 * 4 * 9 / 0.5e12
    assert cost([first, shift, last], prec=L.QD_C128) >= on_pipe
    assert cost([shift, last], prec=L.QD_C128) < 0.3 * on_pipe
    # on a small register a thread's chain of 4 D^2 multiply-adds is what such a launch takes: 25 us
    assert cost([first, shift, last], dims=(3,) * 8, prec=L.QD_C128) >= 25e-6
