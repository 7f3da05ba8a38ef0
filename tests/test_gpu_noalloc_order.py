"""Calls of the allocation-free step that follow each other on one stream without a synchronisation:
each call's set-up kernel rewrites the tiles and scan tables that the call before used, and its
first step has to see them.  A large field is followed by a small one and by the same size with
other parameters, directly and in a captured graph; each against the oracle.

Tolerance: the bound of the allocation-free step's other tests, 1e-12 over tens of steps with
gamma dt / h^4 of order one.
"""
import math

import numpy as np
import pytest

import paper_1911_03386_gb300 as ch
from oracle.oracle import get as get_oracle
from paper_1911_03386_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

H = 2 * math.pi / 128  # gamma dt / h^4 = 0.86 at gamma 0.01, dt 5e-4
CALLS = [(512, 480, 0.01, 5e-4), (33, 40, 0.01, 5e-4), (257, 300, 0.005, 1e-3), (257, 300, 0.01, 2e-4), (16, 17, 0.01, 5e-4),
         (512, 480, 0.005, 5e-4)]


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


@pytest.mark.parametrize("captured", [False, True])
def test_calls_back_to_back_use_their_own_tables(captured):
    torch = pytest.importorskip("torch")
    starts = [wl.random_field(ny, nx, 7 + k, amplitude=0.3, mean=0.1) for k, (nx, ny, _, _) in enumerate(CALLS)]
    fields = [torch.tensor(f, dtype=torch.float64, device="cuda").contiguous() for f in starts]
    nsteps = 3
    # load the kernels before any capture
    warm = torch.tensor(starts[1], dtype=torch.float64, device="cuda").contiguous()
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()

    def step(nx, ny, gamma, dt, field):
        ch.ch_step_field_noalloc(field.data_ptr(), nx, ny, max(nx, ny) * H, gamma, dt, nsteps, stream.cuda_stream)

    step(*CALLS[1], warm)
    stream.synchronize()
    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for call, f in zip(CALLS, fields):
                step(*call, f)
        with torch.cuda.stream(stream):
            graph.replay()
    else:
        for call, f in zip(CALLS, fields):
            step(*call, f)
    stream.synchronize()
    orc = get_oracle()
    for (nx, ny, gamma, dt), start, f in zip(CALLS, starts, fields):
        ref = orc.run(start, max(nx, ny) * H, gamma, dt, nsteps).C
        assert np.max(np.abs(f.cpu().numpy() - ref)) <= 1e-12
