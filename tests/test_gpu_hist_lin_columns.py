"""GPU parity of the linFnComp reduce_by_index where the chunks' folds are combined by rows as well as by bins: few bins,
and chunk counts at the first split (512 chunks of 4096 fp32 or 2048 fp64 elements), one below it and beyond it."""
import numpy as np
import pytest

import oracle
from paper_2310_03568_gb300 import adcomb
from tests._gpu import dev, ensure_lib, host
from tests.test_gpu_hist import keys_oor

pytestmark = pytest.mark.gpu

CHUNK = {np.float32: 4096, np.float64: 2048}


@pytest.fixture(scope="module", autouse=True)
def lib():
    ensure_lib()


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("m,chunks", [(1, 512), (7, 511), (8, 512), (9, 770), (31, 769), (600, 513), (609, 512)])
def test_lin_columns(dt, m, chunks):
    """Functions b +- x with small integer b: every bracketing gives the same bits, only the order counts."""
    g = np.random.default_rng(15)
    n = chunks * CHUNK[dt] - 3
    k = keys_oor(g, n, m)
    v = np.stack([g.integers(-1, 2, n), g.choice([-1, 1], n)], 1).astype(dt)
    h0 = np.stack([g.integers(-3, 4, m), g.choice([-1, 1], m)], 1).astype(dt)
    hb = g.integers(-2, 3, (m, 2)).astype(dt)
    h, saved = adcomb.hist_fwd("lin", m, dev(k), dev(v), dev(h0))
    vb, h0b = adcomb.hist_vjp("lin", m, dev(k), dev(v), dev(h0), h, saved, dev(hb), want_hist0bar=True)
    ref = oracle.hist_fwd("lin", m, k, v, h0)
    vr, h0r = oracle.hist_vjp("lin", m, k, v, hb, h0)
    assert max(np.abs(ref).max(), np.abs(vr).max()) < 2**22  # and so are the partial sums (below 2^24)
    assert np.array_equal(host(h), ref.astype(dt).reshape(m, 2))
    assert np.array_equal(host(vb), vr.astype(dt).reshape(n, 2))
    assert np.array_equal(host(h0b), h0r.astype(dt).reshape(m, 2))
