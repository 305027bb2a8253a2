"""mp_plan_optimal's branch and bound against the oracle's plain search over
every order: the optimum and the offsets of the first optimal order, where
ties are frequent, for 32-bit and 64-bit byte words."""
import numpy as np
import pytest
import torch

import oracle
import tracegen as tg

pytestmark = pytest.mark.gpu


# unit 1 and 64: sums below 2^32 in units; 2^33 + 1 (odd): sums past 2^32 in
# any unit; 2^40: far past 2^32 in bytes, a few units after the division
@pytest.mark.parametrize("unit", (1, 64, (1 << 33) + 1, 1 << 40))
@pytest.mark.parametrize("n", (1, 2, 3, 4, 6, 8))
def test_optimal_ties_and_widths(cuda_lib, unit, n):
    import paper_2203_00448_gb300 as mp

    rng = np.random.default_rng(unit % 1000 + n)
    traces = []
    for k in range(12):
        T = int(rng.integers(1, 9))
        a = rng.integers(0, T, n)
        f = np.minimum(a + rng.integers(1, 6, n), T)
        s = rng.integers(1, (2, 4, 50)[k % 3], n) * unit
        traces.append((T, a, f, s))
    ts = tg.from_arrays(traces)
    off, pk, st = (x.cpu().numpy() for x in mp.plan_optimal(mp.DeviceBatch.from_host(ts, "cuda")))
    assert (st == 0).all()
    for b in range(ts.n_traces):
        T, a, f, s = ts.trace(b)
        opt, o_off = oracle.bruteforce_opt(a, f, s)
        lo, hi = ts.trace_ptr[b], ts.trace_ptr[b + 1]
        assert pk[b] == opt, f"trace {b}"
        assert np.array_equal(off[lo:hi], o_off), f"offsets of trace {b}"
