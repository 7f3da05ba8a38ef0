"""Refusals of the allocation-free step that need no GPU: a grid whose lines do not fit and a step
whose implicit factor is out of range are invalid arguments wherever they are asked for, and are told
before anything is looked up on a device.
"""
import pytest

import paper_1911_03386_gb300 as ch
from paper_1911_03386_gb300 import _build


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()


@pytest.mark.parametrize("nx,ny,L,gamma,dt", [(100000, 8, 6.28, 0.01, 1e-4), (8, 100000, 6.28, 0.01, 1e-4),
                                              (64, 64, 1e-100, 1e200, 1e200)])
def test_refused_before_any_device_work(nx, ny, L, gamma, dt):
    with pytest.raises(ch.ChError) as e:
        ch.ch_step_field_noalloc(16, nx, ny, L, gamma, dt, 1, None)
    assert e.value.code == ch.CH_EINVAL
