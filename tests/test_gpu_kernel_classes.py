"""Which kernel a dense launch runs on, by dimension, size, precision and matrix."""
import math

import numpy as np
import pytest
import torch

from paper_2211_07918_gb300 import qudit as L
from paper_2211_07918_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def name_of(dims, gates, prec, kind=None, tc_min_d=0):
    with L.Register(dims, None, prec) as r:
        L.qd_set_tuning(r.h, L.QD_TUNE_TC_MIN_D, tc_min_d)
        if kind is None:
            plan = L.qd_plan_create(r.h, gates, L.QD_PLAN_NONE)
        else:
            plan = L.qd_plan_create_forms(r.h, gates, [(0, len(gates) - 1)], [kind])
        names = [L.kclass_name(int(c)) for c in L.qd_plan_timings(plan, with_times=False)[2]]
        L.qd_plan_destroy(plan)
    assert len(names) == 1
    return names[0]


def gate(targets, m):
    return [wl.Gate("U", tuple(targets), matrix=m)]


def others(groups):
    """Qudits of about (and at least) that many states."""
    out = []
    while math.prod(out) < groups:
        out.append(max(2, min(64, math.ceil(groups / math.prod(out)))))
    return out


@pytest.mark.parametrize("d", [2, 3, 4, 5, 9, 16, 24, 32])
def test_complex128(d):
    m = np.fft.fft(np.eye(d)) / math.sqrt(d)
    least = {2: 300000, 3: 180000}.get(d, 1)
    assert name_of([d] + others(-(-least // d)), gate([0], m), L.QD_C128) == f"dense_direct_D{d}_tc"
    if d < 4:
        assert name_of([d] + others(least // d // 4), gate([0], m), L.QD_C128) == f"dense_direct_D{d}"
    small = m.copy()
    small[0, 0] *= 2.0 ** -20
    ring = np.eye(d) + np.roll(np.eye(d), 1, axis=1)
    for other in (small, ring) if d > 2 else (small,):
        assert name_of([d] + others(310000 // d), gate([0], other), L.QD_C128) == f"dense_direct_D{d}"
    # a dense part and a phase on another qudit, in one launch
    run = [wl.Gate("DIAG", (1,), matrix=np.exp(1j * np.arange(5)))]
    if d <= 16:
        want = f"dense_table_D{d}_tc"
        assert name_of([d, 5] + others(310000 // d // 5 + 1), gate([0], m) + run, L.QD_C128, L.QD_FORM_DENSE_RUN) == want


@pytest.mark.parametrize("d", [4, 9, 10, 12, 16, 18])
def test_complex64(d):
    m = np.fft.fft(np.eye(d)) / math.sqrt(d)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    between = [300 * sms] + ([560 * sms] if d == 10 else [])
    for groups in [100, 250 * sms // 2] + between + [900 * sms]:
        tc = 10 <= d <= 16 and groups not in between
        dims = [5, d] + others(groups / 5)
        assert name_of(dims, gate([1], m), L.QD_C64) == f"dense_direct_D{d}" + ("_tc" if tc else "")
        assert name_of(dims, gate([1], m), L.QD_C64, tc_min_d=65) == f"dense_direct_D{d}"
    zeros = m.copy()
    zeros[0, 0] = 0
    assert name_of([5, d, 7], gate([1], zeros), L.QD_C64) == f"dense_direct_D{d}"
    run = [wl.Gate("DIAG", (0,), matrix=np.exp(1j * np.arange(5)))]
    if d <= 16:
        assert name_of([5, d, 7], gate([1], m) + run, L.QD_C64, L.QD_FORM_DENSE_RUN) == f"dense_table_D{d}"
