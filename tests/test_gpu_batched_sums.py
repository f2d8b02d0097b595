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


def test_loss_holds_what_a_double_holds():
    """Scan values 2^40, 2^15, 2^-10, -2^40, -2^15 (and zeros between them): the sum is 2^-10, and every partial sum
    fits a double's 53 bits."""
    s = [2.0**40, 0.0, 2.0**15, 0.0, 2.0**-10, 0.0, -(2.0**40), 0.0, -(2.0**15)]
    p = one_value_per_bin(np.diff(np.r_[0.0, s]), "add")
    assert np.array_equal(host(p.scan)[:9], np.float32(s))
    assert host(p.loss)[0] == np.float32(2.0**-10)


@pytest.mark.parametrize("n", [9, 5000])
def test_loss_beyond_the_largest_float(n):
    """Scan values of 2^126 and then their negatives, n of each: the partial sums leave fp32, not a double."""
    big = 2.0**126
    scan = np.r_[np.full(n, big), [0.0], np.full(n, -big)]
    p = one_value_per_bin(np.diff(np.r_[0.0, scan]), "add")
    assert np.array_equal(host(p.scan)[: 2 * n + 1], np.float32(scan))
    assert host(p.loss)[0] == 0.0
