"""GPU: reduce_by_index + vjp whose histogram adjoint is accumulated in place (hist0bar is histbar): the values'
adjoints are gathered from the adjoint as it was.  Integers: exact in every order."""
import numpy as np
import pytest

from paper_2310_03568_gb300 import adcomb
from tests._gpu import dev, ensure_lib, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    ensure_lib()


@pytest.mark.parametrize("n,m", [(0, 7), (3, 100_000), (4_000_003, 1000), (4_000_003, 3_000_001)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_add_hist0bar_in_place(n, m, accumulate):
    g = np.random.default_rng(14)
    k = g.integers(-2, m + 2, n).astype(np.int32)
    hb = g.integers(-50, 51, m).astype(np.float32)
    old = g.integers(-50, 51, n).astype(np.float32)
    hbd = dev(hb)
    vb, h0b = adcomb.hist_vjp("add", m, dev(k), dev(old), None, None, None, hbd, valsbar=dev(old), hist0bar=hbd,
                              accumulate=accumulate)
    inr = (k >= 0) & (k < m)
    want = np.where(inr, hb[np.clip(k, 0, m - 1)], 0) + (old if accumulate else 0)
    assert np.array_equal(host(vb), want)
    assert np.array_equal(host(h0b), 2 * hb if accumulate else hb)
