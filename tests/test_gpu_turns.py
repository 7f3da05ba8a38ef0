"""Cluster-resident FP32 members that take turns in the last wave of a launch: more members than
the device holds at once, stepped in one call, against the same members stepped one step per call
(no turns: a call of one step has nothing to split).  Fields are kept in FP32 between launches,
so both are equal bit for bit, samples included."""
import math

import numpy as np
import pytest

import paper_1911_03386_gb300 as ch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


def run(nx, ny, gamma, members, calls, every):
    with ch.Ensemble.create(nx, ny, 2 * math.pi, gamma, 1e-3, [0.4 * (k % 3) for k in range(members)],
                            11, ch.CH_FP32) as e:
        e.set_tuning(resident=1)  # compensated 256-wide members too
        e.set_sampling(every, 0.0, capacity=16)
        for n in calls:
            e.step(n)
        return [e.field(k) for k in range(members)], [e.series(k, 16) for k in range(members)]


# sizes of the resident form; member counts just above one, two and three waves of it (36 clusters of
# 8 CTAs, 76 of 4 at most; 15 of 8 for compensated 256-wide members, gamma = 0.02); step counts that
# the parts do not divide
@pytest.mark.parametrize("nx,ny,gamma,members,steps", [
    (256, 256, 0.02, 38, 23), (256, 256, 0.02, 75, 17), (256, 128, 0.02, 80, 19), (128, 128, 0.02, 79, 31),
    (128, 256, 0.02, 113, 13), (256, 256, 0.005, 38, 23), (256, 256, 0.005, 75, 17), (256, 128, 0.005, 80, 19)])
def test_turns_equal_single_steps(nx, ny, gamma, members, steps):
    fa, ba = run(nx, ny, gamma, members, [steps], 5)
    fb, bb = run(nx, ny, gamma, members, [1] * steps, 5)
    for k in range(members):
        assert np.array_equal(fa[k], fb[k]), k
        assert len(ba[k]) == (steps + 4) // 5 and np.array_equal(ba[k], bb[k]), k
