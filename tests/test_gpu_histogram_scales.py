"""Histogram bins of values at the ends of the FP32 range, where the bin is decided in FP32 only if
its error bound allows it: counts equal to the oracle's FP64 division for every width that the entry
point takes.  Counts are whole numbers and have no tolerance.
"""
import numpy as np
import pytest

import paper_1911_03386_gb300 as ch
from oracle.oracle import get as get_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__

    __graft_entry__.build()


# bins narrower than the smallest normal FP32 number, of its size, of the bound's absolute part
# (1e-20), near FP32's largest number and beyond it
@pytest.mark.parametrize("lo,w,nbins", [(-3.5e-38, 1e-38, 10), (-1e-39, 3e-40, 40), (0.0, 1e-300, 8), (-4e-19, 1e-19, 9),
                                        (1e-30, 1e-20, 5), (-8e37, 2e37, 9), (0.0, 3e38, 4), (-1e300, 1e299, 33)])
def test_counts_at_every_scale(lo, w, nbins):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(nbins)
    M, T = 257, 33
    hi = lo + nbins * w
    beta = lo + w * rng.uniform(-2, nbins + 2, (M, T))
    beta[:, 1] = lo + w * rng.integers(-1, nbins + 2, M)  # on edges
    beta[0, 2], beta[1, 2], beta[2, 2] = w, -w, 0.0
    beta[3:40, 3] = w * rng.uniform(-1, 1, 37) * 1e-3
    b = torch.tensor(beta, dtype=torch.float64, device="cuda").contiguous()
    out = torch.full((T, nbins + 2), -1, dtype=torch.int64, device="cuda")
    ch.ch_stats_histogram(b.data_ptr(), M, T, T, lo, hi, nbins, out.data_ptr())
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), get_oracle().beta_histogram(beta, lo, hi, nbins))
