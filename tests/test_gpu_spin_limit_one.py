"""GPU: a spin limit of one poll on every scan engine.

Waits run out while bulk copies are in flight; a block then waits for its copies under a limit of their own before it
leaves, so nothing lands in shared memory that has become another block's.  The call reports the timeout (or finishes,
where every first poll happens to succeed), and the next call, with blocks of every kind on the same SMs, is right.
"""
import numpy as np
import pytest

import oracle
from paper_2310_03568_gb300 import adcomb
from tests._gpu import dev, ensure_lib, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    ensure_lib()
    yield
    adcomb.debug_set_scan_engine(0)
    adcomb.set_spin_limit(0)


def exact_inputs(g, op, n):
    """Small integers whose scans and adjoints stay below 2^24: every order of the operations gives the same bits."""
    if op == "add":
        return g.integers(-1, 2, n).astype(np.float32), g.integers(-1, 2, n).astype(np.float32)
    if op == "lin":  # x -> b +- x
        x = np.stack([g.integers(-1, 2, n), g.choice([-1, 1], n)], 1)
        return x.astype(np.float32), g.integers(-1, 2, (n, 2)).astype(np.float32)
    q = int(op[2])  # signed permutation matrices
    x = np.zeros((n, q, q), np.float32)
    perm = np.argsort(g.random((n, q)), axis=1)
    x[np.arange(n)[:, None], np.arange(q)[None, :], perm] = g.choice([-1, 1], (n, q))
    return x.reshape(n, q * q), g.integers(-1, 2, (n, q * q)).astype(np.float32)


@pytest.mark.parametrize("op,engine", [("add", 3), ("lin", 3), ("add", 4), ("lin", 4), ("add", 7), ("lin", 7),
                                       ("mm3", 6), ("mm5", 6)])
def test_one_poll(op, engine):
    g = np.random.default_rng(12)
    n = 60_000 if op in ("mm3", "mm5") else 400_000
    x, yb = exact_inputs(g, op, n)
    xd, ybd = dev(x), dev(yb)
    ref, vref = oracle.scan_fwd(op, x), oracle.scan_vjp(op, x, yb)
    assert max(np.abs(ref).max(), np.abs(vref).max()) < 2**24
    y = dev(ref.astype(np.float32).reshape(x.shape))
    ws = adcomb.Workspace()
    calls = [(lambda: adcomb.scan_fwd(op, xd, ws=ws), ref), (lambda: adcomb.scan_vjp(op, xd, y, ybd, ws=ws), vref)]
    try:
        adcomb.debug_set_scan_engine(engine)
        for call, want in calls:
            adcomb.set_spin_limit(1)
            for _ in range(4):
                call()
            assert adcomb.check_device_error(ws) in (0, 5)
            adcomb.set_spin_limit(0)
            out = host(call())
            assert adcomb.check_device_error(ws) == 0
            assert np.array_equal(out, want.astype(np.float32).reshape(out.shape))
    finally:
        adcomb.set_spin_limit(0)
        adcomb.debug_set_scan_engine(0)
