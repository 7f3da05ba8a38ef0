"""The fixed-point form of the CH_FP64 step (csrc/ch_fixed.cu) against the oracle and the FP64
kernels, at the edges of its segments, bands, panels and classes.

Tolerances: the form holds at least as many bits as FP64 at every stage, so a step's result differs
from the oracle's by the oracle's own rounding (2^-53 of C per step, and the rounding of R' passed
through the solves, at most kappa-scaled cond(I + s D^4) = 1 + 16 s per direction): the bound of the
other FP64 forms, 1e-12 over tens of steps at s of order one, and nsteps 2u (1 + 16 s) max|dC_1| at
large s.
"""
import math

import numpy as np
import pytest

import paper_1911_03386_gb300 as ch
from oracle.oracle import get as get_oracle
from paper_1911_03386_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TWO_PI = 2 * math.pi
SEED = wl.BASE_SEED


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


# segment lengths change at 64 | 65, 128 | 129 (rows) and 256 | 257 (panels), bands at 8 and 16 rows;
# last segments of 1 and S - 1 points, last panels of one column, the smallest and largest lines
SIZES = [(16, 16), (17, 16), (31, 33), (63, 64), (64, 65), (65, 63), (97, 130), (128, 129), (129, 128), (255, 40),
         (256, 257), (257, 24), (511, 18), (513, 20), (16, 512), (24, 513), (1024, 16), (16, 1024), (1023, 17)]


def domain(n, hx=TWO_PI / 128):
    return n * hx


@pytest.mark.parametrize("nx,ny", SIZES)
def test_line_lengths_match_oracle(nx, ny):
    orc = get_oracle()
    L, gamma, dt, nsteps = domain(nx), 0.01, 5e-4, 12
    sx = gamma * dt / (L / nx) ** 4
    sy = gamma * dt / (L / ny) ** 4
    with ch.Ensemble.create(nx, ny, L, gamma, dt, [0.0, 0.3], SEED, ch.CH_FP64) as e:
        first = [e.field(k) for k in range(2)]
        e.step(1)
        one = max(float(np.max(np.abs(e.field(k) - first[k]))) for k in range(2))
        e.step(nsteps - 1)
        tol = 1e-12 + nsteps * 2.0 ** -52 * (1 + 16 * max(sx, sy)) * one
        for k, c0 in enumerate((0.0, 0.3)):
            ref = orc.run(first[k], L, gamma, dt, nsteps)
            assert np.max(np.abs(e.field(k) - ref.C)) <= tol
            W = e.row_solve(k)
            assert np.all(np.isfinite(W))


def test_agrees_with_the_fp64_kernels_in_a_mix():
    # one batch with every class; each member alone gives the same bits
    sizes = [(48, 40), (64, 64), (100, 30), (128, 128), (200, 33), (256, 64), (300, 300), (700, 20)]
    descs = [dict(nx=nx, ny=ny, L=domain(nx), gamma=0.01, dt=5e-4, C0=0.1 * k, seed=SEED, counter_base=10 ** 6 * k)
             for k, (nx, ny) in enumerate(sizes)]
    nsteps = 40
    with ch.Ensemble.batch(descs, ch.CH_FP64) as e, ch.Ensemble.batch(descs, ch.CH_FP64) as old:
        old.set_tuning(split=1)  # the FP64 kernels
        e.step(nsteps)
        old.step(nsteps)
        mix = [e.field(k) for k in range(len(sizes))]
        for k in range(len(sizes)):
            assert np.max(np.abs(mix[k] - old.field(k))) <= 1e-12
        assert np.allclose(e.observables()[0], old.observables()[0], rtol=1e-12, atol=0)
    for k, d in enumerate(descs):
        with ch.Ensemble.batch([d], ch.CH_FP64) as a:
            a.step(nsteps)
            assert np.array_equal(a.field(0), mix[k])


@pytest.mark.parametrize("scale", [1e-70, 1e-30, 1e-6, 0.9, 1.999, 2.0, 3.0])
def test_magnitudes_in_and_out_of_the_scaled_range(scale):
    # 2^-200 <= max|C| < 2 runs in fixed point, the rest in FP64; relative agreement in both
    orc = get_oracle()
    f = scale * np.cos(np.arange(40)[None, :] * 0.3 + np.arange(36)[:, None] * 0.7) * 0.999
    f[3, 5] = scale
    L, gamma, dt, nsteps = domain(40), 0.01, 1e-5, 5
    with ch.Ensemble.create(40, 36, L, gamma, dt, [0.0], SEED, ch.CH_FP64) as e:
        e.set_field(0, f)
        e.step(nsteps)
        ref = orc.run(f, L, gamma, dt, nsteps).C
        assert np.max(np.abs(e.field(0) - ref)) <= 1e-14 * np.max(np.abs(ref))


def test_a_band_out_of_range_beside_others():
    # zeros (a band whose largest |C| has no binary exponent) and large values in some bands only
    orc = get_oracle()
    f = wl.random_field(64, 72, 3, amplitude=0.4)
    f[20:40] = 0.0
    f[50, 7] = 2.5
    L, gamma, dt, nsteps = domain(72), 0.01, 1e-4, 6
    with ch.Ensemble.create(72, 64, L, gamma, dt, [0.0], SEED, ch.CH_FP64) as e:
        e.set_field(0, f)
        e.step(nsteps)
        ref = orc.run(f, L, gamma, dt, nsteps).C
        assert np.max(np.abs(e.field(0) - ref)) <= 1e-13


def test_a_nan_spreads_as_in_the_fp64_kernels():
    with ch.Ensemble.create(96, 80, TWO_PI, 0.01, 1e-3, [0.0, 0.3], SEED, ch.CH_FP64) as e:
        e.step(2)
        ch.ch_set_fault("nan:1")
        try:
            e.step(2)
        finally:
            ch.ch_set_fault(None)
        assert np.all(np.isfinite(e.field(0)))
        assert np.all(np.isnan(e.field(1)))
        with pytest.raises(ch.ChError) as err:
            e.observables()
        assert err.value.code == ch.CH_ENONFINITE


def test_constant_field_stays_and_mass_is_conserved():
    with ch.Ensemble.create(100, 64, TWO_PI, 0.01, 1e-3, [0.0], SEED, ch.CH_FP64) as e:
        e.set_field(0, np.full((64, 100), 0.37))
        e.step(20)
        assert np.array_equal(e.field(0), np.full((64, 100), 0.37))
        f = wl.random_field(64, 100, 5, amplitude=0.5, mean=0.2)
        e.set_field(0, f)
        e.step(200)
        # each point's update rounds at 2^-53 |C| per step, without bias: sqrt(200) 2^-53 on average
        assert abs(np.mean(e.field(0)) - np.mean(f)) <= math.sqrt(200) * 2.0 ** -53
