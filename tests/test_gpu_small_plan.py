"""Batches of few small traces, which one launch plans, and the line beyond
which two launches do: most tensors and steps of its range, empty traces, and
sizes summing to 2^32 and more beside small ones."""
import numpy as np
import pytest

import tracegen as tg

from tests.test_gpu_phases import _check, _trace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,T,traces", ((1, 1, 1), (63, 40, 3), (64, 2048, 5), (64, 2049, 5), (65, 130, 5), (64, 96, 608),
                                        (64, 96, 609)))
@pytest.mark.parametrize("unit", (1, (1 << 27) + 1))
def test_small_traces(cuda_lib, n, T, traces, unit):
    rng = np.random.default_rng(n * 7 + T + traces)
    ts = []
    for k in range(traces):
        m = n if k == 0 else 0 if k == 2 else int(rng.integers(1, n + 1))
        # every third trace with sizes that may sum past 2^32
        ts.append(_trace(rng, m, T, 0.2 if T > 40 else 0.0, unit if k % 3 == 0 else 1, 64, life=min(T, 6)))
    _check(tg.from_arrays(ts))
