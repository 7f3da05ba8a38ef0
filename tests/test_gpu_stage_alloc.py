"""The staging buffer of CH_FP32 field transfers: an ensemble whose device has no room for it converts
on the host with the same values, and a server has it from its creation, so that a run's result is
read back without an allocation.
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


@pytest.mark.parametrize("nx,ny,gamma", [(48, 31, 0.005), (1200, 901, 0.01)])  # plain, compensated
def test_transfers_without_staging(nx, ny, gamma):
    x = np.random.default_rng(nx).uniform(-1, 1, (2, ny, nx))
    got = []
    for fault in (None, "alloc"):
        with ch.Ensemble.create(nx, ny, TWO_PI, gamma, 1e-3, [0.0, 0.1], 3, ch.CH_FP32) as e:
            out = []
            for f in (lambda: e.set_fields_ptr(x.ctypes.data), lambda: e.set_field(1, x[0]), lambda: out.append(e.field(0)),
                      lambda: out.append(e.field(1))):
                ch.ch_set_fault(fault)  # each transfer tries again: all four on the host
                try:
                    f()
                finally:
                    ch.ch_set_fault(None)
            both = np.empty_like(x)
            e.get_fields_ptr(both.ctypes.data)  # staged
            out += list(both)
        got.append(out)
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_server_reads_results_without_allocating():
    run = dict(nx=300, ny=200, L=TWO_PI, gamma=0.005, dt=1e-4, C0=0.2, seed=3, nsteps=5)
    with ch.Server(8 << 20, ch.CH_FP32) as s:
        s.wait(s.submit(**run), 60.0)  # tile tables at their size
        field = np.zeros((200, 300))
        ch.ch_set_fault("alloc:1")  # fires at the next allocation of the library
        try:
            s.wait(s.submit(**run, field_out=field), 60.0)
            with pytest.raises(ch.ChError) as e:  # still armed: nothing was allocated
                ch.Ensemble.create(64, 64, TWO_PI, 0.005, 1e-4, [0.0], 3, ch.CH_FP32)
            assert e.value.code == ch.CH_ENOMEM
        finally:
            ch.ch_set_fault(None)
    with ch.Ensemble.create(300, 200, TWO_PI, 0.005, 1e-4, [0.2], 3, ch.CH_FP32) as e:
        e.step(5)
        assert np.array_equal(e.field(0), field)


def test_failed_staging_allocation_in_server_create():
    # the last of the server's allocations: 8 buffers, its tile tables, then the staging buffer
    for n in range(9, 30):
        ch.ch_set_fault("alloc:%d" % n)
        try:
            ch.Server(8 << 20, ch.CH_FP32).close()
            break  # the fault did not fire: n - 1 allocations in all
        except ch.ChError as e:
            assert e.code == ch.CH_ENOMEM
            last = str(e)
        finally:
            ch.ch_set_fault(None)
    assert "staging" in last
