"""GPU parity: row scans at the edge between one state per unit of 64 rows (up to 1024
units) and one per block, where the min/max forward and one-hot adjoints are exact."""
import numpy as np
import pytest

import oracle
from paper_2310_03568_gb300 import adcomb
from tests._gpu import dev, ensure_lib, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    ensure_lib()


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("d", [2, 11, 32])
@pytest.mark.parametrize("n", [63, 64, 65, 64 * 31 + 1, 64 * 1024 - 1, 64 * 1024, 64 * 1024 + 1])
def test_vscan_max_units(n, d, dt):
    g = np.random.default_rng(61)
    x = ((g.integers(0, 32, (n, d)) - 16) / 4.0).astype(dt)
    y = adcomb.vscan_fwd("max", dev(x))
    assert np.array_equal(host(y), oracle.vscan_fwd("max", x).astype(dt))
    yb = (g.integers(0, 4, (n, d)) - 1).astype(dt)  # whole numbers: sums exact below 2^24
    xb = adcomb.vscan_vjp("max", dev(x), y, dev(yb))
    assert np.array_equal(host(xb), oracle.vscan_vjp("max", x, yb).astype(dt))
