"""GPU: the streaming scans in forms that share something -- a vjp that writes over ybar, two scans at once on two
streams, a captured graph replayed on new data.  Integers whose results stay below 2^24: exact in every order."""
import numpy as np
import pytest
import torch

import oracle
from paper_2310_03568_gb300 import adcomb
from tests._gpu import dev, ensure_lib, host

pytestmark = pytest.mark.gpu

N = 1_200_007  # above 3 MB an array for the pairs and the scalars


@pytest.fixture(scope="module", autouse=True)
def lib():
    ensure_lib()


def inputs(g, op, dt=np.float32):
    if op == "add":
        return g.integers(-1, 2, N).astype(dt), g.integers(-1, 2, N).astype(dt)
    if op == "mul":
        return g.choice([-1, 1], N).astype(dt), g.integers(-1, 2, N).astype(dt)
    if op == "max":
        return g.integers(-1000, 1000, N).astype(dt), g.integers(-1, 2, N).astype(dt)
    x = np.stack([g.integers(-1, 2, N), g.choice([-1, 1], N)], 1).astype(dt)  # lin: x -> b +- x
    return x, g.integers(-1, 2, (N, 2)).astype(dt)


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("op", ["add", "mul", "max", "lin"])
def test_vjp_over_ybar(op, dt):
    """One input array (joint fold and store warps), two, and three (split warps in fp32, joint in fp64)."""
    g = np.random.default_rng(16)
    x, yb = inputs(g, op, dt)
    ref = oracle.scan_vjp(op, x, yb)
    assert np.abs(ref).max() < 2**24
    y = dev(oracle.scan_fwd(op, x).astype(dt).reshape(x.shape))
    for accumulate in (False, True):
        b = dev(yb)
        adcomb.scan_vjp(op, dev(x), y, b, xbar=b, accumulate=accumulate)
        want = ref.reshape(yb.shape) + (yb if accumulate else 0)
        assert np.array_equal(host(b), want.astype(dt))


def test_two_streams_at_once():
    """Each scan wants a whole SM per block; neither may wait for a block of the other's that is not running."""
    g = np.random.default_rng(17)
    jobs = []
    for op in ("add", "lin"):
        x, yb = inputs(g, op)
        jobs.append((op, dev(x), dev(yb), oracle.scan_fwd(op, x), oracle.scan_vjp(op, x, yb), torch.cuda.Stream(),
                     adcomb.Workspace()))
    out = []
    torch.cuda.synchronize()
    for _ in range(10):
        for op, x, yb, _, _, s, ws in jobs:
            with torch.cuda.stream(s):
                y = adcomb.scan_fwd(op, x, ws=ws)
                out.append((op, y, adcomb.scan_vjp(op, x, y, yb, ws=ws)))
    torch.cuda.synchronize()
    for (op, y, xb), (_, _, _, yr, xr, _, _) in zip(out, jobs * 10):
        assert np.array_equal(host(y), yr.astype(np.float32).reshape(y.shape)), op
        assert np.array_equal(host(xb), xr.astype(np.float32).reshape(xb.shape)), op
    for *_, ws in jobs:
        assert adcomb.check_device_error(ws) == 0


def test_captured_graph_on_new_data():
    g = np.random.default_rng(18)
    x, yb = inputs(g, "lin")
    xd, ybd, xb, ws = dev(x), dev(yb), torch.empty(N, 2, device="cuda"), adcomb.Workspace()
    y = adcomb.scan_fwd("lin", xd, ws=ws)
    adcomb.scan_vjp("lin", xd, y, ybd, xbar=xb, ws=ws)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        adcomb.scan_fwd("lin", xd, y, ws=ws)
        adcomb.scan_vjp("lin", xd, y, ybd, xbar=xb, ws=ws)
    for _ in range(2):
        x, yb = inputs(g, "lin")
        xd.copy_(dev(x))
        ybd.copy_(dev(yb))
        graph.replay()
        assert np.array_equal(host(y), oracle.scan_fwd("lin", x).astype(np.float32).reshape(N, 2))
        assert np.array_equal(host(xb), oracle.scan_vjp("lin", x, yb).astype(np.float32).reshape(N, 2))
    assert adcomb.check_device_error(ws) == 0
