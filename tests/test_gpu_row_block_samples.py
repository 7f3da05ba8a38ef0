"""Samples of the transposed-block row form (tuning row_seg = 1), whose CTAs have nx / 32 warps: the
exact sums of F and dF/dt need a buffer that does not shrink with the warps.  The sums are exact, so
they are those of every other form, bit for bit.
"""
import math

import numpy as np
import pytest

import paper_1911_03386_gb300 as ch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("nx", [32, 64, 96, 128, 160, 512])
@pytest.mark.parametrize("ny", [33, 64])
def test_samples_of_narrow_block_rows(nx, ny):
    rows = []
    for t in (dict(split=0, row_seg=1, resident=-1), dict(split=1, resident=-1)):
        with ch.Ensemble.create(nx, ny, nx * 2 * math.pi / 128, 0.01, 5e-4, [0.0, 0.3], 11, ch.CH_FP32) as e:
            e.set_tuning(**t)
            e.set_sampling(1, 0.0, 4)
            e.step(1)
            rows.append([e.series(k, 4) for k in range(2)])
    assert np.array_equal(rows[0], rows[1])
    assert np.all(np.isfinite(rows[0]))
