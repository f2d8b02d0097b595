"""GPU: the streaming scans' carried roundings.  A constant coefficient gives every
tile the same product, so a tile's error is repeated by every tile behind it:
rounded at each multiplication, c^n over 1e6 elements is off by about 1e-3.
Carried, each of the T <= 250 tiles adds at most three roundings (the published
product and two combines), and the last tile at most 16 + 8 + 2 x 255 of its own
(row, levels, unnormalised products), each of 2^-24 relative: below 1e-4."""
import numpy as np
import pytest

from paper_2310_03568_gb300 import adcomb
from tests._gpu import dev, ensure_lib, host

pytestmark = pytest.mark.gpu
N, C, TOL = 1_000_003, np.float32(1.00001), 1e-4


@pytest.fixture(scope="module", autouse=True)
def lib():
    ensure_lib()


def powers(n):
    return np.float64(C) ** np.arange(n)


@pytest.mark.parametrize("op", ["mul", "lin"])
def test_products_of_a_constant(op):
    p = powers(N + 1)
    if op == "mul":
        y = host(adcomb.scan_fwd("mul", dev(np.full(N, C, np.float32))))
        assert np.max(np.abs(y / p[1:] - 1)) <= TOL
        return
    x = np.zeros((N, 2), np.float32)
    x[:, 1], x[0, 0] = C, 1
    y = host(adcomb.scan_fwd("lin", dev(x)))
    assert np.max(np.abs(y[:, 0] / p[:-1] - 1)) <= TOL
    assert np.max(np.abs(y[:, 1] / p[1:] - 1)) <= TOL


@pytest.mark.parametrize("op", ["mul", "lin"])
def test_adjoints_of_a_constant(op):
    """Only the last output has an adjoint: lambda_i = c^(n - 1 - i)."""
    lam = powers(N)[::-1]
    if op == "mul":
        x, yb = np.full(N, C, np.float32), np.zeros(N, np.float32)
        y = np.ones(N, np.float32)  # xbar_i = y_{i-1} lambda_i
        yb[-1] = 1
        xb = host(adcomb.scan_vjp("mul", dev(x), dev(y), dev(yb)))
    else:
        x, yb = np.zeros((N, 2), np.float32), np.zeros((N, 2), np.float32)
        x[:, 1], yb[-1, 0] = C, 1
        xb = host(adcomb.scan_vjp("lin", dev(x), dev(np.zeros((N, 2), np.float32)), dev(yb)))[:, 0]
    assert np.max(np.abs(xb / lam - 1)) <= TOL


@pytest.mark.parametrize("op", ["add", "mul", "sop", "lin"])
def test_infinities_stay_infinite(op):
    """One infinite element: outputs before it are finite, all others are not."""
    w = 2 if op in ("lin", "sop") else 1
    x = np.full((N, w), 0.5, np.float32)
    at = N // 2
    x[at] = np.inf
    y = host(adcomb.scan_fwd(op, dev(x if w == 2 else x[:, 0]))).reshape(N, w)
    # (for *, 0.5^i underflows to 0 long before, and 0 * inf is NaN)
    assert np.isfinite(y[:at]).all() and not np.isfinite(y[at:]).any()


@pytest.mark.parametrize("direction", ["fwd", "vjp"])
def test_small_elements_after_a_large_prefix(direction):
    """2^25 (whose unit in the last place is 4), zeros to the end of the 8192-element
    tile, then halves: every row's, tile's and running sum is a multiple of 16 below
    2^26, so exact, and a result rounds once, by at most 2."""
    n = 128 * 8192
    x = np.full(n, 0.5, np.float32)
    x[:8192] = 0
    x[0] = 2.0**25
    ref = np.cumsum(x.astype(np.float64))
    if direction == "fwd":
        got = host(adcomb.scan_fwd("add", dev(x)))
    else:
        r = dev(x[::-1].copy())
        got = host(adcomb.scan_vjp("add", r, r, r))[::-1]
    assert np.max(np.abs(got - ref)) <= 2
