"""Field transfers of CH_FP32 handles, converted on the device in pieces of 32 MiB: values that need
rounding, in fields that end inside a piece, and compensated members (hi + lo pairs); and the
allocation-free step on the grids where its line form changes, against the oracle.

Transfers are exact by definition: a plain member stores the nearest FP32 value, a compensated one
hi = fl(x) and lo = fl(x - hi), read back as their FP64 sum.  The allocation-free step holds at least
FP64's bits at every stage: 1e-12 over tens of steps at s of order one, as for the handles.
"""
import math

import numpy as np
import pytest

import paper_1911_03386_gb300 as ch
from oracle.oracle import get as get_oracle
from paper_1911_03386_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TWO_PI = 2 * math.pi


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("nx,ny,gamma", [(48, 31, 0.01), (2048, 2048, 1e-7), (2051, 2049, 1e-7), (1200, 1201, 0.01)])
def test_fp32_transfers_are_exact(nx, ny, gamma):
    x = np.random.default_rng(nx).uniform(-1, 1, (ny, nx))
    comp = gamma * 1e-3 / (TWO_PI / nx) ** 4 > 16 or gamma * 1e-3 / (TWO_PI / ny) ** 4 > 16
    hi = x.astype(np.float32)
    want = hi.astype(np.float64) + (x - hi).astype(np.float32).astype(np.float64) if comp else hi.astype(np.float64)
    with ch.Ensemble.create(nx, ny, TWO_PI, gamma, 1e-3, [0.0, 0.1], 3, ch.CH_FP32) as e:
        other = e.field(0)
        e.set_field(1, x)
        assert np.array_equal(e.field(1), want)
        assert np.array_equal(e.field(0), other)
        both = np.stack([x, -x])
        e.set_fields_ptr(both.ctypes.data)
        got = np.empty_like(both)
        e.get_fields_ptr(got.ctypes.data)
        assert np.array_equal(got[0], want) and np.array_equal(got[1], -want)


@pytest.mark.parametrize("nx,ny", [(16, 16), (65, 64), (64, 129), (257, 40), (512, 96), (31, 513), (1024, 16), (1000, 33)])
def test_noalloc_lines_match_oracle(nx, ny):
    torch = pytest.importorskip("torch")
    L, gamma, dt, nsteps = nx * TWO_PI / 128, 0.01, 5e-4, 12
    start = wl.random_field(ny, nx, 5, amplitude=0.3, mean=0.1)
    C = torch.tensor(start, dtype=torch.float64, device="cuda").contiguous()
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    ch.ch_step_field_noalloc(C.data_ptr(), nx, ny, L, gamma, dt, nsteps, st.cuda_stream)
    st.synchronize()
    orc = get_oracle()
    first = start.copy()
    orc.step(first, L, gamma, dt)
    s = gamma * dt / min(L / nx, L / ny) ** 4
    tol = 1e-12 + nsteps * 2.0 ** -52 * (1 + 16 * s) * np.max(np.abs(first - start))
    assert np.max(np.abs(C.cpu().numpy() - orc.run(start, L, gamma, dt, nsteps).C)) <= tol
