"""Which kernel places a trace, over the lines of the rules that choose it (the
routes are counted in a test build of the library), and its results there
against the oracle."""
import numpy as np
import pytest

import tracegen as tg

from tests.test_gpu_phases import _check, _far_trace, _trace

pytestmark = pytest.mark.gpu


def _linked(rng, n, sizes=64, life=3):
    """One component of n tensors without long-lived ones: each overlaps the next."""
    a = np.arange(n)
    return n + life + 1, a, a + rng.integers(2, life + 1, size=n), rng.integers(1, sizes + 1, size=n) * 256


def _small(rng):
    return _trace(rng, 30, 40, 0.0, 64, 1 << 14)


def _plans(ts, routes):
    """Routes of one call per policy of the planner by size, and by breadth."""
    import paper_2203_00448_gb300 as mp

    db = mp.DeviceBatch.from_host(ts, "cuda")
    got = []
    for fn in (mp.plan_and_validate, mp.plan_greedy_by_size, mp.plan_greedy_by_breadth):
        for policy in ("first", "best"):
            fn(db, policy)
            got.append(routes())
    assert all(g == got[0] for g in got[:4]), got
    return got[0], got[4], got[5]


# (traces, members of the component, route): 34 traces and 310 are on either side of what the phases hold at once
@pytest.mark.parametrize("traces,n,route", ((34, 65, "walk"), (34, 128, "walk"), (34, 129, "phases"), (310, 65, "walk"),
                                            (34, 200, "phases"), (310, 129, "walk"), (310, 1023, "walk"),
                                            (310, 1024, "walk"), (310, 1025, "phases")))
def test_chains(routes, traces, n, route):
    rng = np.random.default_rng(n + traces)
    ts = tg.from_arrays([_linked(rng, n if k % 16 == 0 else 30, (3, 1 << 12)[k // 16 % 2]) for k in range(traces)])
    big = (traces + 15) // 16
    size, _, _ = _plans(ts, routes)
    assert size == {"first": traces - big, route: big}
    _check(ts)


# a step's tensors: windows of 2.8 times as many positions on average, on either side of the rule's lines for the
# average (48 a step: 134 positions) and the sum (38 a step: 106, 40,432 for 380 members; twice that with 1,824 traces)
@pytest.mark.parametrize("traces,steps,per_step,route", ((34, 10, 16, "phases"), (310, 10, 38, "walk"), (310, 10, 39, "phases"),
                                                         (310, 5, 52, "walk"), (310, 5, 53, "phases"),
                                                         (1824, 10, 48, "walk"), (1824, 10, 49, "phases"),
                                                         (1823, 10, 48, "phases")))
def test_wide_windows(routes, traces, steps, per_step, route):
    rng = np.random.default_rng(per_step + traces)
    ts = []
    for k in range(traces):
        if k % 100:
            ts.append(_small(rng))
            continue
        a = np.repeat(np.arange(steps), per_step)  # each lives two steps
        ts.append((steps + 2, a, a + 2, rng.integers(1, 1 << 10, len(a)) * 64))
    big = (traces + 99) // 100
    ts = tg.from_arrays(ts)
    size, _, _ = _plans(ts, routes)
    assert size == {"first": traces - big, route: big}
    _check(ts)


def test_long_lived_members_are_not_walked(routes):
    rng = np.random.default_rng(1)
    ts = [_small(rng) for _ in range(320)]
    T, a, f, s = _linked(rng, 200)
    f[50] = a[50] + 32  # the longest a short-lived tensor lives
    ts[3] = (T, a, f, s)
    T, a, f, s = _linked(rng, 200)
    f[50] = a[50] + 33
    ts[7] = (T, a, f, s)
    ts = tg.from_arrays(ts)
    size, _, _ = _plans(ts, routes)
    assert size == {"first": 318, "walk": 1, "phases": 1}
    _check(ts)


@pytest.mark.parametrize("T,route", ((400, "walk"), (401, "phases")))
def test_sparse_batches_do_not_walk(routes, T, route):
    """Fewer than three tensors in four steps (by the longest trace): the kernel without the walk."""
    rng = np.random.default_rng(2)
    _, a, f, s = _linked(rng, 300)
    ts = tg.from_arrays([_small(rng) for _ in range(310)] + [(T, a, f, s)])
    size, _, _ = _plans(ts, routes)
    assert size == {"first": 310, route: 1}
    _check(ts)


# the most tensors the phases take, with the most steps; and the most of a launch that has 256 threads a trace
@pytest.mark.parametrize("traces,n,T,route", ((34, 4080, 4248, "phases"), (34, 4080, 4249, "general"), (34, 4081, 300, "general"),
                                              (160, 2048, 2400, "phases"), (160, 2049, 2400, "phases"),
                                              (160, 4080, 4248, "phases")))
def test_phases_limits(routes, traces, n, T, route):
    rng = np.random.default_rng(n + T)
    ts = [_small(rng) for _ in range(traces)]
    for k in (1, traces - 1):
        ts[k] = _trace(rng, n, T, 0.05, 64, 1 << 14, full_span=k > 1)
    ts = tg.from_arrays(ts)
    size, first, best = _plans(ts, routes)
    assert size == {"first": traces - 2, route: 2}
    other = {"phases": "breadth-phases", "general": "breadth-tensor"}[route]
    assert first == best and first[other] == 2 if other == "breadth-tensor" else first[other] >= 2
    _check(ts)


@pytest.mark.parametrize("traces,T,route", ((160, 5466, "walk"), (160, 5467, "general"), (33, 5466, "general")))
def test_long_traces_without_phases(routes, traces, T, route):
    """Traces past the phases' limits, and too long on average for a launch that
    takes the others: walked by 128 threads in a larger batch, with few tensors a
    step or few traces left to the general path."""
    rng = np.random.default_rng(T)
    ts = [_linked(rng, 1020) for _ in range(traces - 1)]
    _, a, f, s = _trace(rng, 4100, 5000, 0.0, 64, 1 << 14, life=2)
    ts.append((T, a, f, s))
    ts = tg.from_arrays(ts)
    size, _, _ = _plans(ts, routes)
    assert size == {"first": 1, route: traces - 1}
    _check(ts)


@pytest.mark.parametrize("traces", (40, 160))
def test_a_long_trace_among_ordinary_ones(routes, traces):
    """One trace past the phases' limits leaves them to the others."""
    rng = np.random.default_rng(traces)
    ts = [_small(rng) for _ in range(traces)]
    for k in (0, 5, 9):
        ts[k] = _trace(rng, 500, 600, 0.05, 64, 1 << 14, full_span=k > 0)
    ts[3] = _trace(rng, 2000, 20000, 0.0, 64, 1 << 14)  # steps
    ts[4] = _trace(rng, 5000, 4000, 0.02, 64, 1 << 14, full_span=True)  # tensors
    ts = tg.from_arrays(ts)
    size, first, best = _plans(ts, routes)
    assert size == {"first": traces - 4, "phases": 3, "general": 1}
    assert first == best and first["breadth-phases"] >= 3
    _check(ts)


def test_phases_leave_what_they_cannot_take(routes):
    """Sums of 2^32 units, too many long-lived tensors, a long chain beside one: the general path."""
    rng = np.random.default_rng(8)
    ts = [_small(rng) for _ in range(36)]
    ok = lambda: _trace(rng, 1200, 1300, 0.0, 64, 1 << 10)
    for k, wide, longs, link in ((0, 0, 0, False), (1, 1, 0, False), (2, 0, 768, False), (3, 0, 769, False), (4, 0, 0, True),
                                 (5, 0, 1, True)):
        T, a, f, s = ok()
        if link:
            a, f = np.minimum(np.arange(len(a)), T - 3), np.minimum(np.arange(len(a)) + 2, T)
        a[-1], f[-1] = 0, 2 if link and not longs else T  # held together by it
        if longs > 1:
            a[:longs - 1] = rng.integers(0, 300, longs - 1)
            f[:longs - 1] = a[:longs - 1] + rng.integers(33, 800, longs - 1)
            a[longs - 1:-1] = rng.integers(900, T - 5, len(a) - longs)
            f[longs - 1:-1] = a[longs - 1:-1] + 1
        if wide:
            s[0] = (1 << 40) + 1
        ts[k] = (T, a, f, s)
    ts = tg.from_arrays(ts)
    size, _, _ = _plans(ts, routes)
    assert size == {"first": 30, "phases": 3, "general": 3}
    _check(ts)


@pytest.mark.parametrize("traces,n,first,best", ((34, 64, "comp", "comp"), (34, 65, "phases", "phases"),
                                                 (913, 128, "tensor", "phases"), (913, 129, "phases", "phases"),
                                                 (1825, 128, "tensor", "tensor")))
def test_breadth_chains(routes, traces, n, first, best):
    rng = np.random.default_rng(n + traces)
    ts = [_small(rng) for _ in range(traces)]
    for k in (0, traces - 1):
        ts[k] = _linked(rng, n)
    if n == 64:
        ts[0] = (2 * n + ts[0][0], *ts[0][1:])  # steps, the component kernel's scratch
        ts[traces - 1] = ts[0]
    ts = tg.from_arrays(ts)
    got = _plans(ts, routes)[1:]
    assert got == tuple({"breadth-comp": traces} if r == "comp" else {"breadth-comp": traces - 2, "breadth-" + r: 2}
                        for r in (first, best))
    _check(ts)


# tensors of a step: on either side of the lines for a batch that the phases hold at once, and for a larger one
@pytest.mark.parametrize("traces,per_step,route", ((34, 101, "phases"), (34, 102, "tensor"), (310, 7, "phases"),
                                                   (310, 8, "tensor")))
def test_breadth_dense(routes, traces, per_step, route):
    rng = np.random.default_rng(per_step + traces)
    ts = [_small(rng) for _ in range(traces)]
    a = np.repeat(np.arange(40), per_step)
    f = a + 1
    f[::per_step] += 1  # links its step to the next
    ts[5] = (41, a, f, rng.integers(1, 1 << 10, len(a)) * 64)
    ts = tg.from_arrays(ts)
    got = _plans(ts, routes)[1:]
    assert got[0] == got[1] == {"breadth-comp": traces - 1, "breadth-" + route: 1}
    _check(ts)


@pytest.mark.parametrize("T", (400, 401))
def test_breadth_tensor_by_tensor_in_large_batches(routes, T):
    """More traces than the phases' launch holds at once, some of which it refuses:
    by a launch of their own with many tensors a step, else by the phases' launch."""
    rng = np.random.default_rng(3)
    ts = [_small(rng) for _ in range(400)]
    for k in (0, 199, 399):
        _, a, f, s = _trace(rng, 300, 400, 0.05, 1, 1 << 10, full_span=True)
        s[0] = (1 << 40) + 1
        ts[k] = (T, a, f, s)
    ts[7] = _trace(rng, 300, T, 0.05, 1, 1 << 10, full_span=True)
    ts = tg.from_arrays(ts)
    got = _plans(ts, routes)[1:]
    assert got[0] == got[1] == {"breadth-comp": 396, "breadth-phases": 1, "breadth-tensor": 3}
    _check(ts)


def _spanned(rng, n, longs):
    """One chain of n tensors, `longs` of which span it instead."""
    T, a, f, s = _linked(rng, n, 1 << 12)
    far = rng.permutation(n)[:longs]
    a[far], f[far] = 0, T
    return T, a, f, s


@pytest.mark.parametrize("kind,n,first,best", (("long-tail", 5000, "phases", "flow"), ("full-span", 6001, "phases", "phases"),
                                               ("crowded-steps", 7000, "phases", "phases"), ("wide-sums", 4500, "flow", "flow"),
                                               ("short-only", 5000, "flow", "flow"), ("all-long", 4200, "flow", "flow"),
                                               ("chain-10", 2000, "flow", "flow"), ("chain-30", 2000, "phases", "phases"),
                                               ("dense", 2000, "flow", "flow")))
def test_large_traces(routes, kind, n, first, best):
    import paper_2203_00448_gb300 as mp

    rng = np.random.default_rng(n + len(kind))
    if kind.startswith("chain"):
        t = _spanned(rng, n, int(kind[6:]))
    elif kind == "dense":  # few gaps between the chains of short-lived tensors: one warp would walk nearly all
        t = _far_trace(rng, n, n // 5, "long-tail")
    else:
        t = _far_trace(rng, n, n // 2 + 100, kind)
    empty = np.zeros(0, np.int64)
    ts = tg.from_arrays([t, (5, empty, empty, empty)])
    db = mp.DeviceBatch.from_host(ts, "cuda")
    for policy, route in (("first", first), ("best", best)):
        for fn in (mp.plan_and_validate, mp.plan_greedy_by_size):
            fn(db, policy)
            assert routes() == {"grid-" + route: 2}, policy
    if n <= 5000:
        _check(ts)
