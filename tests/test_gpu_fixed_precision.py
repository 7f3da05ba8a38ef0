"""Precision of the fixed-point form of the CH_FP64 step (csrc/ch_fixed.cu): its error and that of
the FP64 kernels (tuning split = 1), both against the same steps in extended precision (numpy
longdouble, at least 64 significant bits), on grids of every aspect ratio.

Tolerances: the form has to be no less precise than the FP64 kernels.  Both errors are sums of many
roundings of about the same size, so the root mean squares over a field agree to a few per cent and
the largest ones to a factor of two: 1.25 and 2 times the FP64 kernels' error.
"""
import math

import numpy as np
import pytest

import paper_1911_03386_gb300 as ch
from oracle.oracle import get as get_oracle

pytestmark = pytest.mark.gpu

TWO_PI = 2 * math.pi
LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


def laplacian(f, hx, hy):
    return ((np.roll(f, -1, 1) - 2 * f + np.roll(f, 1, 1)) / hx ** 2
            + (np.roll(f, -1, 0) - 2 * f + np.roll(f, 1, 0)) / hy ** 2)


def solve_rows(R, s, coefficients=None):
    """(I + s D^4)^-1 along axis 1, periodic (or the recurrences of given p1, p2, over c): D^4 = (z - 2 + 1/z)^2 factored into a forward and a
    backward recurrence with the characteristic root a inside the unit circle, a + 1/a = 2 + i/sqrt(s)."""
    if coefficients:
        p1, p2, c = coefficients
    else:
        s = LD(s)
        w = np.clongdouble(2) + np.clongdouble(1j) / np.sqrt(s)
        d = np.sqrt(w * w - 4)
        a = 2 / (w + d if abs(w + d) >= abs(w - d) else w - d)
        p1, p2, c = 2 * a.real, -(a.real ** 2 + a.imag ** 2), s / (a.real ** 2 + a.imag ** 2)
    n, pre = R.shape[1], int(50 / -math.log(math.sqrt(float(-p2)))) + 50  # the wrap has decayed below 1e-21

    def forward(r):
        r = np.ascontiguousarray(r.T)
        x = y = np.zeros(r.shape[1], LD)
        out = np.empty_like(r)
        for q in range(-pre, n):
            x, y = r[q % n] + p1 * x + p2 * y, x
            if q >= 0:
                out[q] = x
        return out.T

    return forward(forward(R)[:, ::-1])[:, ::-1] / c


def steps_extended(f, L, gamma, dt, n):
    ny, nx = f.shape
    C, hx, hy, g, dt = f.astype(LD), LD(L) / nx, LD(L) / ny, LD(gamma), LD(dt)
    for _ in range(n):
        R = dt * laplacian(C * C * C - C - g * laplacian(C, hx, hy), hx, hy)
        W = solve_rows(R, g * dt / hx ** 4)
        C = C + solve_rows(W.T, g * dt / hy ** 4).T
    return C


def noise(ny, nx):
    return 0.1 * (2 * np.random.default_rng(nx * 5003 + ny).random((ny, nx)) - 1)


def separated(ny, nx):
    x, y = np.arange(nx) * TWO_PI / nx, np.arange(ny) * TWO_PI / ny
    f = np.cos(2 * x)[None, :] * np.cos(3 * y + 0.4)[:, None] + 0.7 * np.sin(x[None, :] - 4 * y[:, None])
    return np.tanh(2.5 * f)


def errors(f, L, gamma, dt, nsteps):
    ny, nx = f.shape
    ref = steps_extended(f, L, gamma, dt, nsteps)
    out = []
    for t in ({}, dict(split=1)):
        with ch.Ensemble.create(nx, ny, L, gamma, dt, [0.0], 1, ch.CH_FP64) as e:
            if t:
                e.set_tuning(**t)
            e.set_field(0, f)
            e.step(nsteps)
            d = np.abs(e.field(0) - ref)
            out.append((float(np.sqrt(np.mean(d * d))), float(np.max(d))))
    return out


# gamma dt / h^4 of the closer spacing: 220, 420, 3200 | 0.86 at a spacing of 2 pi / 128 | wide, 420
GRIDS = [(33, 512, TWO_PI), (17, 600, TWO_PI), (17, 1000, TWO_PI), (140, 513, 513 * TWO_PI / 128),
         (200, 1024, 1024 * TWO_PI / 128), (97, 100, TWO_PI), (600, 17, TWO_PI)]


@pytest.mark.parametrize("start", [noise, separated])
@pytest.mark.parametrize("nx,ny,L", GRIDS)
def test_no_less_precise_than_fp64_at_any_aspect_ratio(nx, ny, L, start):
    fixed, fp64 = errors(start(ny, nx), L, 0.01, 5e-4, 2)
    assert fixed != fp64  # another form ran
    assert fixed[0] <= 1.25 * fp64[0]
    assert fixed[1] <= 2.0 * fp64[1]


def step_with_library_coefficients(f, L, gamma, dt):
    """One step of an n x n field in extended precision with the library's own FP64 coefficients, so
    that a form's error is its rounding alone (at large s the coefficients' is as large)."""
    n = f.shape[0]
    h2 = (L / n) ** 2
    c, p1, p2, _ = ch.ch_penta_factor(gamma * dt / h2 ** 2)
    C, a, b = f.astype(LD), LD(1 - 2 * gamma / h2 - 2 * gamma / h2), LD(gamma / h2)

    def around(g):
        return np.roll(g, 1, 1) + np.roll(g, -1, 1) + np.roll(g, 1, 0) + np.roll(g, -1, 0)

    mu = C * (C * C - a) - b * around(C)
    W = solve_rows(around(mu) - 4 * mu, None, (LD(p1), LD(p2), LD(1)))
    return C + LD(dt / (h2 * c * c)) * solve_rows(W.T, None, (LD(p1), LD(p2), LD(1))).T


@pytest.mark.parametrize("s", [2e4, 4e4, 8e4])  # gain 2^7.4, 2^7.8, 2^8.3
@pytest.mark.parametrize("n", [64, 128])
def test_no_less_precise_than_fp64_at_large_s(n, s):
    # noise in 8 rows and a hundredth of it elsewhere, so that one band's scale is the whole field's;
    # the root mean square over 24 fields: each has a few independent long waves, so the two pooled
    # errors of equal size differ by a few per cent
    gamma, seeds = 0.01, 24
    dt = s * (TWO_PI / n) ** 4 / gamma
    f = np.stack([2 * np.random.default_rng(k).random((n, n)) - 1 for k in range(seeds)])
    f[:, 8:] *= 0.01
    total = []
    for t in ({}, dict(split=1)):
        with ch.Ensemble.create(n, n, TWO_PI, gamma, dt, [0.0] * seeds, 1, ch.CH_FP64) as e:
            if t:
                e.set_tuning(**t)
            e.set_fields_ptr(f.ctypes.data)
            e.step(1)
            total.append([e.field(k) for k in range(seeds)])
    ref = [step_with_library_coefficients(g, TWO_PI, gamma, dt) for g in f]
    fixed, fp64 = (sum(float(np.mean((g - r) ** 2)) for g, r in zip(out, ref)) for out in total)
    assert math.sqrt(fixed / fp64) <= 1.05


@pytest.mark.parametrize("scale", [1.9, 2.1, 3.9, 4.1, 7.9])  # the scale's exponents end at 2, 4 and 8
@pytest.mark.parametrize("nx,ny", [(64, 64), (100, 70), (48, 96)])
@pytest.mark.parametrize("start", [noise, separated])
def test_no_less_precise_than_fp64_at_large_values(nx, ny, start, scale):
    f = start(ny, nx)
    f *= scale / np.max(np.abs(f))
    fixed, fp64 = errors(f, nx * TWO_PI / 128, 0.01, 2e-6, 2)
    assert fixed != fp64
    assert fixed[0] <= 1.25 * fp64[0]
    assert fixed[1] <= 2.0 * fp64[1]


# the active part: a quarter of the box, some columns, some rows
@pytest.mark.parametrize("part", [(slice(0, 0.5), slice(0, 0.5)), (slice(0, 1), slice(0.25, 0.5)), (slice(0.5, 0.75), slice(0, 1))])
@pytest.mark.parametrize("nx,ny,s", [(128, 128, 0.9), (256, 200, 0.9), (130, 97, 0.5), (64, 64, 0.05), (600, 48, 10.0)])
def test_quiet_regions_keep_their_own_precision(nx, ny, s, part):
    # 1e-12 of the rest: relative error there against the FP64 kernels'.  Both forms carry the active
    # part's tail there in FP64 with a relative error that grows by a rounding per point, along one
    # recurrence (the FP64 kernels) or in segments and their matrices' powers: factors of 2 and 4 for that
    L = TWO_PI
    dt = s * (L / max(nx, ny)) ** 4 / 0.01
    rows, cols = (slice(round(p.start * n), round(p.stop * n)) for p, n in zip(part, (ny, nx)))
    f = 1e-12 * (2 * np.random.default_rng(nx).random((ny, nx)) - 1)
    f[rows, cols] = separated(ny, nx)[rows, cols]
    ref = steps_extended(f, L, 0.01, dt, 1)
    quiet = np.abs(ref) < 1e-10
    assert np.any(quiet)
    rel = []
    for t in ({}, dict(split=1)):
        with ch.Ensemble.create(nx, ny, L, 0.01, dt, [0.0], 1, ch.CH_FP64) as e:
            if t:
                e.set_tuning(**t)
            e.set_field(0, f)
            e.step(1)
            r = np.abs(e.field(0) - ref)[quiet] / 1e-12
            rel.append((float(np.sqrt(np.mean(r * r))), float(np.max(r))))
    assert rel[0][0] <= 2.0 * rel[1][0]
    assert rel[0][1] <= 4.0 * rel[1][1]


@pytest.mark.parametrize("scale", [0.9, 2.5, 7.0])
def test_samples_at_large_values(scale):
    # F and dF/dt against the FP64 kernels: both round sums of 4096 terms of one sign
    f = separated(64, 64)
    f *= scale / np.max(np.abs(f))
    out = []
    for t in ({}, dict(split=1)):
        with ch.Ensemble.create(64, 64, TWO_PI, 0.01, 1e-6, [0.0], 1, ch.CH_FP64) as e:
            if t:
                e.set_tuning(**t)
            e.set_field(0, f)
            F, D, _ = e.observables()
            out.append((F[0], D[0]))
    for a, b in zip(*out):
        assert abs(a - b) <= 64 * 2.0 ** -53 * abs(b)


@pytest.mark.parametrize("scale", [0.9, 2.5, 7.0, 9.0])
@pytest.mark.parametrize("n", [64, 128])  # tiled, cluster-resident
def test_fp32_samples_at_large_values(n, scale):
    # the same sums of CH_FP32 fields against the oracle's FP64 ones, n^2 terms of one sign each: its
    # n^2 roundings
    f = separated(n, n)
    f *= scale / np.max(np.abs(f))
    with ch.Ensemble.create(n, n, TWO_PI, 0.01, 1e-6, [0.0], 1, ch.CH_FP32) as e:
        e.set_field(0, f)
        F, D, _ = e.observables()
        want = get_oracle().field_observables(e.field(0), TWO_PI, 0.01)
    for a, b in zip((F[0], D[0]), want):
        assert abs(a - b) <= n * n * 2.0 ** -53 * abs(b)


@pytest.mark.parametrize("nx,ny", [(33, 512), (17, 600)])
def test_allocation_free_step_of_tall_grids(nx, ny):
    # its stated agreement with the FP64 kernels: 1e-13
    torch = pytest.importorskip("torch")
    f = noise(ny, nx)
    with ch.Ensemble.create(nx, ny, TWO_PI, 0.01, 5e-4, [0.0], 1, ch.CH_FP64) as e:
        e.set_tuning(split=1)
        e.set_field(0, f)
        e.step(2)
        want = e.field(0)
    C = torch.tensor(f, dtype=torch.float64, device="cuda").contiguous()
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    ch.ch_step_field_noalloc(C.data_ptr(), nx, ny, TWO_PI, 0.01, 5e-4, 2, st.cuda_stream)
    st.synchronize()
    assert np.max(np.abs(C.cpu().numpy() - want)) <= 1e-13
