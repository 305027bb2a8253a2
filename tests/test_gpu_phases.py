"""Traces placed in phases (runs of short-lived tensors between long-lived ones)
against the oracle, by size and by breadth, where the path can go wrong: sizes
around its sort lengths and limits, no or only long-lived tensors, equal and odd
sizes, many tensors at one step, runs larger than a batch of insertions, and
traces it has to leave to the general path."""
import numpy as np
import pytest
import torch

import oracle
import tracegen as tg

pytestmark = pytest.mark.gpu


def _trace(rng, n, T, long_share, unit, distinct, life=4, full_span=False, bunched=False):
    a = rng.integers(0, 3 if bunched else T, n)
    f = a + rng.integers(1, life + 1, n)
    far = rng.random(n) < long_share
    if full_span:
        a = np.where(far, 0, a)
        f = np.where(far, T, f)
    else:
        f = np.where(far, a + rng.integers(30, max(31, T // 2) + 1, n), f)
    return T, a, np.minimum(f, T), rng.integers(1, distinct + 1, n) * unit


def _check(ts):
    import paper_2203_00448_gb300 as mp

    db = mp.DeviceBatch.from_host(ts, "cuda")
    o_prof, o_lb, _ = oracle.live_profile(ts)
    for policy, pol in (("first", oracle.FIT_FIRST), ("best", oracle.FIT_BEST)):
        o_off, o_pk, o_st = oracle.plan_greedy_by_size(ts, pol)
        r = mp.plan_and_validate(db, policy)
        off, pk, st = mp.plan_greedy_by_size(db, policy)
        assert r.status.cpu().numpy().tolist() == o_st.tolist() == st.cpu().numpy().tolist()
        assert np.array_equal(off.cpu().numpy(), o_off), policy
        assert np.array_equal(r.offsets.cpu().numpy(), o_off), policy
        assert np.array_equal(pk.cpu().numpy(), o_pk) and np.array_equal(r.plan_peak.cpu().numpy(), o_pk)
        assert np.array_equal(r.profile.cpu().numpy(), o_prof)
        assert np.array_equal(r.peak_lb.cpu().numpy(), o_lb)
        assert (r.verdict == 1).all() and (r.conflict == -1).all()
        b_off, b_pk, b_st = (x.cpu().numpy() for x in mp.plan_greedy_by_breadth(db, policy))
        p_off, p_pk, p_st = oracle.plan_greedy_by_breadth(ts, pol)
        assert b_st.tolist() == p_st.tolist()
        assert np.array_equal(b_off, p_off), f"breadth {policy}"
        assert np.array_equal(b_pk, p_pk)


# 33 traces and more keep the batch off the grid-wide planner
@pytest.mark.parametrize("n", (66, 511, 512, 513, 1025, 2049))
@pytest.mark.parametrize("unit", (1, 4096))
def test_phases_sizes(cuda_lib, n, unit):
    rng = np.random.default_rng(n + unit)
    traces = []
    for k in range(34):
        m = n if k < 4 else int(rng.integers(1, n + 1))
        traces.append(_trace(rng, m, int(m * (0.4, 1.0, 2.0)[k % 3]) + 40, (0.02, 0.1, 0.0, 0.3)[k % 4], unit,
                             (4, 1 << 20)[k % 2], full_span=k % 5 == 0, bunched=k % 11 == 7))
    _check(tg.from_arrays(traces))


@pytest.mark.parametrize("case", ("largest", "too-many-tensors", "too-many-long", "all-long", "wide-sums",
                                  "dense-short"))
def test_phases_limits(cuda_lib, case):
    rng = np.random.default_rng(len(case))
    traces = [_trace(rng, 50, 100, 0.1, 64, 1 << 14) for _ in range(33)]
    for full in (False, True):
        if case == "largest":  # the most tensors that fit the shared memory, and the most steps with them
            traces.append(_trace(rng, 4080, 4248, 0.05, 64, 1 << 16, full_span=full))
        elif case == "too-many-tensors":  # past the path's limit: the general path
            traces.append(_trace(rng, 4081, 3000, 0.03, 64, 1 << 16, full_span=full))
        elif case == "too-many-long":  # 768 fit, more are left to the general path
            for nl in (768, 769):
                T, a, f, s = _trace(rng, 1000, 1200, 0.0, 64, 1 << 10)
                a[:nl] = rng.integers(0, 300, nl)
                f[:nl] = a[:nl] + rng.integers(33, 800, nl)
                traces.append((T, a, f, s))
        elif case == "all-long":
            T, a, f, s = _trace(rng, 300, 2000, 1.0, 64, 50)
            traces.append((T, a, np.minimum(np.maximum(f, a + 33), T), s))
        elif case == "wide-sums":  # sums just below and above 2^32 units
            for extra in (-1, 0, 1):
                T, a, f, s = _trace(rng, 400, 500, 0.1, 1, 1 << 20, full_span=full)
                s[0] = (1 << 32) - int(s[1:].sum()) + extra
                traces.append((T, a, f, s))
        else:  # every short-lived tensor in one chain, windows past 64 positions
            traces.append(_trace(rng, 1500, 300, 0.02, 64, 1 << 12, life=30, full_span=full))
    _check(tg.from_arrays(traces))


@pytest.mark.parametrize("kind", ("long", "chain"))
def test_phases_refuse_late(cuda_lib, kind):
    """Every trace of the batch is refused only once its long-lived tensors'
    ranks are written, in the shared memory that the general path then clears:
    too many of them, or a chain of over 1,024 positions beside some."""
    rng = np.random.default_rng(len(kind))
    traces = []
    for k in range(40):
        n = 1100 + 7 * k
        if kind == "long":
            T, a, f, s = _trace(rng, n, 1200, 0.0, 64, 1 << 10)
            nl = 769 + k
            a[-nl:] = rng.integers(0, 300, nl)
            f[-nl:] = a[-nl:] + rng.integers(33, 800, nl)
        else:
            T, a, f, s = _trace(rng, n, 220, 0.02, 64, 1 << 10, life=20, full_span=True)
        traces.append((T, a, f, s))
    ts = tg.from_arrays(traces)
    for _ in range(4):
        _check(ts)


def _far_trace(rng, n, T, kind):
    a = rng.integers(0, T, n)
    f = a + rng.integers(1, 6, n)
    s = rng.integers(1, 1 << 16, n) * 64
    far = rng.random(n) < 0.05
    if kind == "long-tail":
        f = np.where(far, a + rng.integers(100, T // 2 + 1, n), f)
    elif kind == "full-span":  # groups of one lifetime, few sizes
        a, f = np.where(far, 0, a), np.where(far, T, f)
        s = rng.choice([64, 4096, 1 << 20], n)
    elif kind == "crowded-steps":  # over kEdges tensors just before a long one's start, chains past kNear neighbours
        a[: 1500] = rng.integers(10, 14, 1500)
        f = a + rng.integers(1, 9, n)
        f[:4] = a[:4] + 60
        a[4:8], f[4:8] = 16, T
        a[8:308], f[8:308] = 0, T  # enough that phases pay
    elif kind == "wide-sums":  # past 2^32 units: the dataflow
        s[0], s[1] = (1 << 35) + 1, 1
    elif kind == "short-only":
        pass
    elif kind == "all-long":
        f = a + 33 + rng.integers(0, 40, n)
        far[:] = True
    return T, a, np.minimum(f, T), s


@pytest.mark.parametrize("kind,n", (("long-tail", 5000), ("long-tail", 20000), ("full-span", 6001), ("crowded-steps", 7000),
                                    ("wide-sums", 4500), ("short-only", 23000), ("short-only", 24000),
                                    ("all-long", 4200), ("mixed", 9000), ("phased", 9000),
                                    ("empty-first", 6000)))
def test_large_traces_in_phases(cuda_lib, kind, n):
    """One large trace per SM (batches of a few, past what one CTA prepares in
    its shared memory), and those left to the grid-wide dataflow."""
    import paper_2203_00448_gb300 as mp

    rng = np.random.default_rng(n + len(kind))
    kinds = {"mixed": ("long-tail", "full-span", "wide-sums", "short-only"),
             "phased": ("long-tail", "full-span", "long-tail"), "empty-first": ("full-span",)}.get(kind, (kind,))
    traces = [_far_trace(rng, n, n // 2 + 100, k) for k in kinds]
    if kind == "empty-first":  # no record of their own to load, and none before them
        none = np.zeros(0, np.int64)
        traces = [(10, none, none, none), (0, none, none, none)] + traces
    if kind in ("mixed", "phased"):
        traces += [(10, np.zeros(0, np.int64), np.zeros(0, np.int64), np.zeros(0, np.int64)),
                   (9, np.array([0, 3]), np.array([4, 2]), np.array([8, 8])),  # free <= alloc
                   _far_trace(rng, 300, 200, "short-only")]
    ts = tg.from_arrays(traces)
    db = mp.DeviceBatch.from_host(ts, "cuda")
    o_prof, o_lb, _ = oracle.live_profile(ts)
    for policy, pol in (("first", oracle.FIT_FIRST), ("best", oracle.FIT_BEST)):
        o_off, o_pk, o_st = oracle.plan_greedy_by_size(ts, pol)
        r = mp.plan_and_validate(db, policy)
        off, pk, st = mp.plan_greedy_by_size(db, policy)
        st, rst = st.cpu().numpy(), r.status.cpu().numpy()
        assert st.tolist() == o_st.tolist() == rst.tolist()
        for b in np.flatnonzero(o_st == 0):
            lo, hi = ts.trace_ptr[b], ts.trace_ptr[b + 1]
            assert np.array_equal(off[lo:hi].cpu().numpy(), o_off[lo:hi]), (policy, b)
            assert np.array_equal(r.offsets[lo:hi].cpu().numpy(), o_off[lo:hi]), (policy, b)
            assert int(pk[b]) == o_pk[b] == int(r.plan_peak[b]) and int(r.verdict[b]) == 1
            plo, phi = ts.profile_ptr[b], ts.profile_ptr[b + 1]
            assert np.array_equal(r.profile[plo:phi].cpu().numpy(), o_prof[plo:phi]) and int(r.peak_lb[b]) == o_lb[b]
