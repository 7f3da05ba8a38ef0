"""Samples of a CH_FP64 run whose values leave the scaled range of the fixed-point form (|C| >= 8):
its CTAs have 64 to 256 threads, depending on the other runs of the launch, and F, dF/dt and beta
must not.
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


def run(sizes, f, dt):
    descs = [dict(nx=nx, ny=ny, L=nx * TWO_PI / 128, gamma=0.01, dt=dt, C0=0.0, seed=3, counter_base=10 ** 6 * k)
             for k, (nx, ny) in enumerate(sizes)]
    with ch.Ensemble.batch(descs, ch.CH_FP64) as e:
        e.set_field(0, f)
        e.set_sampling(1, 0.0, 8)
        e.step(4)
        F, D, B = e.observables()
        return e.series(0, 8), (F[0], D[0], B[0]), e.field(0)


@pytest.mark.parametrize("scale,dt", [(1.0, 1e-5), (4.0, 1e-6)])
@pytest.mark.parametrize("nx,ny", [(64, 60), (128, 100)])
def test_samples_out_of_range_do_not_depend_on_company(nx, ny, scale, dt):
    x, y = np.arange(nx) * TWO_PI / nx, np.arange(ny) * TWO_PI / ny
    f = 2.6 * np.cos(2 * x)[None, :] * np.cos(y + 0.3)[:, None] + 0.5 * np.sin(5 * x[None, :] + 3 * y[:, None])
    f *= scale
    alone = run([(nx, ny)], f, dt)
    assert (np.max(np.abs(alone[2])) > 8) == (scale > 1)  # still in or out of range
    # its class in CTAs of its own size; beside other classes in CTAs of 256 threads
    for company in ([(nx, ny)] * 40, [(nx, ny), (256, 64), (48, 40), (100, 90)]):
        got = run(company, f, dt)
        assert np.array_equal(got[0], alone[0])
        assert got[1] == alone[1]
        assert np.array_equal(got[2], alone[2])
