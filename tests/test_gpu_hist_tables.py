"""GPU parity at the edges of the reduce_by_index `*` table forms: the reduction of
the blocks' partial rows by 16-byte words (m >= 16,384 and a multiple of the word),
the vjp with its coefficient table in shared memory (64 KB < table <= 200 KB and
n >= 64 m) and both neighbours; and the batched problem on keys and values whose
16-byte boundaries differ."""
import numpy as np
import pytest
import torch

import oracle
from paper_2310_03568_gb300 import adcomb, batched as B, synth
from tests._gpu import dev, ensure_lib, host
from tests._tol import assert_tol, rtol_for
from tests.test_gpu_batched import check_problem, oracle_reference, small_workload
from tests.test_gpu_hist import bin_partial_products, bin_stats, keys_oor

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    ensure_lib()
    yield
    adcomb.debug_force_hist_strategy(-1)


# m at the first and last table of each form (in elements of the type), one past it, and
# a remainder; n at 64 m, one below, and with ragged ends
TABLES = [(np.float32, 16_384, 64 * 16_384), (np.float32, 16_385, 64 * 16_385), (np.float32, 16_388, 64 * 16_388 - 1),
          (np.float32, 20_002, 64 * 20_002 + 3), (np.float32, 51_200, 64 * 51_200 + 1),
          (np.float32, 51_201, 64 * 51_201), (np.float64, 8_192, 64 * 8_192), (np.float64, 8_193, 64 * 8_193 + 2),
          (np.float64, 16_386, 64 * 16_386), (np.float64, 25_600, 64 * 25_600 + 1),
          (np.float64, 25_601, 64 * 25_601)]


@pytest.mark.parametrize("dt,m,n", TABLES)
def test_hist_mul_tables(dt, m, n):
    g = np.random.default_rng(26)
    rtol = rtol_for(dt)
    adcomb.debug_force_hist_strategy(1 if m * np.dtype(dt).itemsize <= 200 * 1024 else -1)  # per block
    k = keys_oor(g, n, m)
    v = np.exp(g.uniform(-1, 1, n) * 3.0 / np.sqrt(n / m)).astype(dt)
    first = np.unique(np.where((k >= 0) & (k < m), k, m), return_index=True)
    zeros = first[1][(first[0] < m) & (first[0] % 5 == 0)]  # one zero in every fifth bin, two in the first bins
    v[zeros] = 0
    v[np.nonzero(k == 0)[0][:2]] = 0
    h0 = synth.uniform(g, m, 0.5, 1.5, dt)
    h, saved = adcomb.hist_fwd("mul", m, dev(k), dev(v), dev(h0))
    pop, _ = bin_stats(k, v, m)
    part = bin_partial_products(k, v, m)
    pmax = part * np.abs(h0)
    assert_tol("hist * fwd", host(h), oracle.hist_fwd("mul", m, k, v, h0), pop + 1, pmax, rtol)
    nz_r, p_r = oracle.hist_mul_lifted(m, k, v)
    sv = host(saved)
    assert np.array_equal(sv[: 4 * m].view(np.int32), nz_r.astype(np.int32))
    off = ((4 * m + 15) // 16) * 16
    assert_tol("hist * p", sv[off: off + m * np.dtype(dt).itemsize].view(dt), p_r, pop, part, rtol)
    hb = synth.normal(g, m, dt)
    vr, _ = oracle.hist_vjp("mul", m, k, v, hb, h0)
    inr = (k >= 0) & (k < m)
    kc = np.clip(k, 0, m - 1)
    scale = np.where(inr, pmax[kc] * np.abs(hb[kc]) /
                     np.where(v != 0, np.minimum(np.abs(v.astype(np.float64)), 1), 1), 0)
    nj = np.where(inr, pop[kc], 1)
    old = synth.normal(g, n, dt)
    for acc in (False, True):
        vb, _ = adcomb.hist_vjp("mul", m, dev(k), dev(v), dev(h0), h, saved, dev(hb),
                                valsbar=dev(old) if acc else None, want_hist0bar=False, accumulate=acc)
        ref = vr + old if acc else vr
        assert_tol("hist * vjp", host(vb), ref, nj, np.maximum(scale, np.abs(old)) if acc else scale, rtol)


@pytest.mark.parametrize("chunk", [333, 1 << 14])
@pytest.mark.parametrize("shift", [1, 2, 3])
def test_batched_misaligned_keys(chunk, shift):
    """Keys `shift` elements off the values' 16-byte boundaries: element by element."""
    desc, keys, vals = B.layout(small_workload(seed=36, count=24))
    p = B.BatchedHistScan(desc, keys, vals, chunk=chunk)
    buf = torch.empty(p.keys.numel() + shift, dtype=p.keys.dtype, device=p.keys.device)
    buf[shift:] = p.keys
    p.keys = buf[shift:]
    p.forward()
    p.backward()
    torch.cuda.synchronize()
    check_problem(p, desc, keys, vals, oracle_reference(desc, keys, vals))
