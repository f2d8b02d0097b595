"""GPU parity of the streaming scan engine (hook 7 forces it at every size; it is the automatic choice
from 3 MB per input array on): edges of its rows, segments and tiles, many rounds of tiles, accumulation, in-place
forwards, and its bounded waits."""
import numpy as np
import pytest

import oracle
from paper_2310_03568_gb300 import adcomb, synth
from tests._gpu import dev, ensure_lib, host
from tests._tol import assert_tol, rtol_for, suffix_max
from tests.test_gpu_scan import check_scan, make_x

pytestmark = pytest.mark.gpu

WORDS = {"add": 1, "mul": 1, "max": 1, "lin": 2, "sop": 2, "mm2": 4}


@pytest.fixture(scope="module", autouse=True)
def lib():
    ensure_lib()
    adcomb.debug_set_scan_engine(7)
    yield
    adcomb.debug_set_scan_engine(0)


def edge_sizes(op, dt):
    """Around one row (64 / 128 bytes), one warp's segment and one tile (8 segments), forward and vjp shapes."""
    e = WORDS[op] * np.dtype(dt).itemsize
    out = {1, 2, 3}
    for row in (64, 128):
        for k in (1, 32, 8 * 32, 3 * 8 * 32):
            out |= {max(1, k * row // e + d) for d in (-1, 0, 1)}
    return sorted(out)


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("op", ["add", "mul", "lin", "sop", "mm2"])
def test_stream_edges(op, dt):
    g = np.random.default_rng(51 + len(op))
    for n in edge_sizes(op, dt):
        x = make_x(g, op, n, dt)
        check_scan(op, x, synth.normal(g, x.shape, dt), dt)
    x = make_x(g, op, edge_sizes(op, dt)[-1], dt)
    check_scan(op, x, synth.normal(g, x.shape, dt), dt, accumulate=True)


@pytest.mark.parametrize("op,dt,n", [("add", np.float32, 5_000_011), ("mul", np.float64, 3_000_001),
                                     ("lin", np.float32, 3_000_001), ("sop", np.float64, 1_500_007),
                                     ("mm2", np.float32, 1_500_007)])
def test_stream_many_rounds(op, dt, n):
    """Several tiles per block (152 blocks, tiles of 16 or 32 KB per array) and a ragged last one."""
    g = np.random.default_rng(52)
    x = make_x(g, op, n, dt)
    check_scan(op, x, synth.normal(g, x.shape, dt), dt)


@pytest.mark.parametrize("dt", [np.float32, np.float64])
def test_stream_minmax(dt):
    g = np.random.default_rng(53)
    for n in edge_sizes("max", dt) + [2_000_003]:
        for op in ("min", "max"):
            x = ((g.integers(0, 64, n) - 32) / 8.0).astype(dt)
            x[g.random(n) < 0.01] = np.nan
            x[0] = 1.0
            yb = g.integers(-3, 4, n).astype(dt)
            old = g.integers(-3, 4, n).astype(dt)
            xd = dev(x)
            y = adcomb.scan_fwd(op, xd)
            assert np.array_equal(host(y), oracle.scan_fwd(op, x).astype(dt))
            xb = adcomb.scan_vjp(op, xd, y, dev(yb), xbar=dev(old), accumulate=True)
            ref = oracle.scan_vjp(op, x, yb) + old
            assert_tol(f"scan {op} vjp", host(xb), ref, n - np.arange(n), suffix_max(yb) + np.abs(old), rtol_for(dt))


def test_stream_nan_first_and_in_place():
    x = np.arange(20_000, dtype=np.float32)
    x[0] = np.nan
    assert np.isnan(host(adcomb.scan_fwd("max", dev(x)))).all()
    v = np.ones(1_000_003, np.float32)
    d = dev(v)
    adcomb.scan_fwd("add", d, d)  # y is x: a tile is staged before it is overwritten
    assert np.array_equal(host(d), np.arange(1, v.shape[0] + 1, dtype=np.float32))


@pytest.mark.parametrize("op,stall", [("add", 3), ("lin", 0), ("mm2", 17)])
def test_stream_stall_times_out(op, stall):
    """A tile that never publishes: later tiles' waits run out, the error is reported, the context survives."""
    g = np.random.default_rng(8)
    n = 400_000
    x = synth.scan_values(g, op, n) if op != "add" else synth.uniform(g, n, -1, 1)
    yb = synth.normal(g, x.shape)
    xd, ybd = dev(x), dev(yb)
    y = adcomb.scan_fwd(op, xd)
    ws = adcomb.Workspace()
    calls = [lambda: adcomb.scan_fwd(op, xd, ws=ws)]
    if op != "mm2":
        calls.append(lambda: adcomb.scan_vjp(op, xd, y, ybd, ws=ws))
    for call in calls:
        try:
            adcomb.set_spin_limit(2000)
            adcomb.debug_set_stall_tile(stall)
            call()
            assert adcomb.check_device_error(ws) == 5
        finally:
            adcomb.debug_set_stall_tile(-1)
            adcomb.set_spin_limit(0)
        call()
        assert adcomb.check_device_error(ws) == 0
    ref = oracle.scan_fwd(op, x)
    np.testing.assert_allclose(host(adcomb.scan_fwd(op, xd, ws=ws)).reshape(ref.shape), ref, rtol=1e-3, atol=1e-2)
