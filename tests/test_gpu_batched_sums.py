"""GPU: precision of the batched hist -> +-scan -> sum pipeline's own sums, on values chosen so that the exact result
is known."""
import numpy as np
import pytest
import torch

from paper_2310_03568_gb300 import batched as B
from tests._gpu import ensure_lib, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    ensure_lib()


def one_value_per_bin(h, op):
    h = np.asarray(h, np.float32)
    desc = B.make_table([h.shape[0]], [h.shape[0]], [op])
    p = B.BatchedHistScan(desc, np.arange(h.shape[0], dtype=np.int32), h)
    p.forward()
    torch.cuda.synchronize()
    return p


@pytest.mark.parametrize("op", ["add", "max"])
def test_scan_adds_the_prefix_once_per_bin(op):
    """Ones after 2^24: each result is the exact sum, rounded (half a unit, 1, at most)."""
    p = one_value_per_bin([2.0**24] + [0.0] * 7 + [1.0] * 8, op)
    assert np.abs(host(p.scan)[:16].astype(np.float64) - (2.0**24 + np.r_[[0] * 8, 1:9])).max() <= 1
