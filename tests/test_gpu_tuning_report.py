"""The report of ch_get_tuning passed back to ch_set_tuning keeps the fixed-point form of CH_FP64
members, which has no field of its own.  The forms round differently, so equal fields after some steps show which one ran.
"""
import math

import numpy as np
import pytest

import paper_1911_03386_gb300 as ch

pytestmark = pytest.mark.gpu

TWO_PI = 2 * math.pi


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


def advance(descs, tuning=None, report_back=False):
    with ch.Ensemble.batch(descs, ch.CH_FP64) as e:
        if tuning:
            e.set_tuning(**tuning)
        report = e.tuning()
        if report_back:
            e.set_tuning(**report)
            assert e.tuning() == report
        e.step(20)
        return report, [e.field(k) for k in range(len(descs))]


@pytest.mark.parametrize("sizes", [[(64, 48)], [(256, 256)], [(64, 1024)], [(96, 80), (1040, 24), (40, 33)]])
def test_report_passed_back_keeps_the_fixed_point_form(sizes):
    descs = [dict(nx=nx, ny=ny, L=max(nx, ny) * TWO_PI / 128, gamma=0.01, dt=5e-4, C0=0.1, seed=5, counter_base=10 ** 6 * k)
             for k, (nx, ny) in enumerate(sizes)]
    report, want = advance(descs)
    _, back = advance(descs, report_back=True)
    assert all(np.array_equal(a, b) for a, b in zip(want, back))
    fp64_report, fp64 = advance(descs, tuning=dict(split=1))
    assert fp64_report["split"] == 1 and fp64_report["threads"] == 512
    assert not np.array_equal(want[0], fp64[0])
