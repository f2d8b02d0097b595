"""GPU: a bounded wait that runs out inside reduce_by_index is a status, and nothing is read or written by it.

The kernels after the wait take bins and element numbers from scratch memory that the giving-up block was to fill.
The scratch is filled with ones here, so what was never written is neither a bin of any table nor an element, and a
kernel that believed it would leave its arrays.  The waits run out through the fault-injection hook: one chunk's (one
tile's) data never comes.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2310_03568_gb300 import adcomb, synth
from tests._gpu import dev, ensure_lib, host

pytestmark = pytest.mark.gpu

TIMEOUT = 5


@pytest.fixture(scope="module", autouse=True)
def lib():
    ensure_lib()
    yield
    adcomb.debug_set_stall_tile(-1)
    adcomb.set_spin_limit(0)


def ones_workspace(kind, op, n, m):
    ws = adcomb.Workspace()
    ws.buf = torch.full((adcomb.workspace_bytes(kind, op, torch.float32, n, m),), 255, dtype=torch.uint8,
                        device="cuda")
    return ws


def stalled(call, ws, tile, limit):
    try:
        adcomb.set_spin_limit(limit)
        adcomb.debug_set_stall_tile(tile)
        call()
        assert adcomb.check_device_error(ws) == TIMEOUT
    finally:
        adcomb.debug_set_stall_tile(-1)
        adcomb.set_spin_limit(0)


@pytest.mark.parametrize("stall", [0, 300, 609])
@pytest.mark.parametrize("op", ["add", "mul", "min", "max"])
def test_partitioned_chunk_that_never_comes(op, stall):
    g = np.random.default_rng(11)
    m = 1 << 19
    n = 610 * 8192 + 5  # two and some chunks per block; chunk 610 is loaded by plain loads
    keys = g.integers(0, m, n).astype(np.int32)
    v = synth.uniform(g, n, 0.5, 2.0)
    kd, vd = dev(keys), dev(v)
    ws = ones_workspace("hist", op, n, m)
    hist = torch.full((m,), 7.0, device="cuda")
    saved = torch.full((max(adcomb.saved_bytes("hist", op, torch.float32, n, m), 16),), 255, dtype=torch.uint8,
                       device="cuda")
    stalled(lambda: adcomb.hist_fwd(op, m, kd, vd, None, hist, saved, ws=ws), ws, stall, 500)
    empty = {"add": 0.0, "mul": 1.0, "min": np.inf, "max": -np.inf}[op]
    assert (host(hist) == empty).all()  # every bin empty: no element was touched
    if op in ("min", "max"):
        assert (host(saved.view(torch.int32))[:m] == n).all()  # and none selected
    elif op == "mul":
        assert (host(saved.view(torch.int32))[:m] == 0).all()
    # the context is intact and the same workspace works again
    adcomb.hist_fwd(op, m, kd, vd, None, hist, saved, ws=ws)
    assert adcomb.check_device_error(ws) == 0
    ref = oracle.hist_fwd(op, m, keys, v)
    # about 10 positive values a bin, at most some 40: 40 roundings of 2^-24
    np.testing.assert_allclose(host(hist), ref[0] if isinstance(ref, tuple) else ref, rtol=2.5e-6, atol=0)


@pytest.mark.parametrize("m,forced", [(5000, -1), (100, 2)], ids=["two-pass", "one-pass"])
def test_sorted_path_without_offsets(m, forced):
    """linFnComp through the radix sort: the scan of the counts times out, so no element has a destination."""
    g = np.random.default_rng(13)
    n = 300_000
    keys = g.integers(0, m, n).astype(np.int32)
    v = np.stack([g.standard_normal(n), g.uniform(0.95, 1.05, n)], 1).astype(np.float32)
    hb = g.standard_normal((m, 2)).astype(np.float32)
    kd, vd, hbd = dev(keys), dev(v), dev(hb)
    try:
        adcomb.debug_force_hist_strategy(forced)
        ws = ones_workspace("hist", "lin", n, m)
        hist = torch.full((m, 2), 7.0, device="cuda")
        saved = torch.full((adcomb.saved_bytes("hist", "lin", torch.float32, n, m),), 255, dtype=torch.uint8,
                           device="cuda")
        stalled(lambda: adcomb.hist_fwd("lin", m, kd, vd, None, hist, saved, ws=ws), ws, 0, 2000)  # the counts are two tiles or more
        assert (host(hist) == np.array([0.0, 1.0], np.float32)).all()
        # the residuals may be followed: no element has a bin
        vb, _ = adcomb.hist_vjp("lin", m, kd, vd, None, hist, saved, hbd, ws=ws)
        assert adcomb.check_device_error(ws) == 0
        assert (host(vb) == 0).all()
        adcomb.hist_fwd("lin", m, kd, vd, None, hist, saved, ws=ws)
        assert adcomb.check_device_error(ws) == 0
        np.testing.assert_allclose(host(hist), oracle.hist_fwd("lin", m, keys, v).reshape(m, 2), rtol=1e-3, atol=1e-2)
    finally:
        adcomb.debug_force_hist_strategy(-1)
