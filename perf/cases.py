"""The work a user of this framework has it do, as cases that can be timed.

A case is one call path (``op``) over one batch of allocation traces
(``kind`` and its sizes):

op        path       profile, greedy_by_size plan and its validation in one pass (plan_and_validate)
          plan       the greedy_by_size plan alone (plan_greedy_by_size)
          profile    the live-bytes profile alone (live_profile)
          validate   a plan in hand checked pair by pair, and its peak (validate_plan, peak)
          breadth    the greedy-by-breadth plan (plan_greedy_by_breadth)
          optimal    the exact optimum of tiny traces (plan_optimal)
          host       the whole path from pinned host buffers to host buffers (HostPath)
kind      random     lifetimes of a few steps, sizes log-uniform 64 B .. 1 MiB; ``ragged`` traces differ in length
          chain      a ResNet-50-shaped chain of ops: equal activations that live 1 to 3 steps, residuals 3 to 4
          longtail   5% of the tensors live for 100 steps up to half of the trace, sizes up to 64 MiB
          seq2seq    activations and per-token state of a serving step, 2% of the tensors live throughout
          tiny       at most 10 tensors over 6 steps, as the exact optimum takes them

All results are integers and are compared exactly.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2203_00448_gb300 as mp

# ResNet-50's stage shapes (channels, height = width).
STAGES = np.array([[64, 112], [256, 56], [512, 28], [1024, 14], [2048, 7]], dtype=np.int64)


def listed():
    return [
        # one captured trace planned at load time or for a new input shape: latency counts
        {"name": "path-single", "op": "path", "kind": "random", "traces": 1, "n": 64, "T": 128, "ragged": False,
         "policy": "first"},
        # one vision model's inference graph
        {"name": "path-chain", "op": "path", "kind": "chain", "traces": 1, "n": 374, "T": 160, "ragged": False,
         "policy": "first"},
        # an offline sweep: every trace of a corpus planned and checked in one call
        {"name": "path-batch", "op": "path", "kind": "random", "traces": 4096, "n": 512, "T": 1024, "ragged": False,
         "policy": "first"},
        # a service's ordinary batch of models of all lengths, odd ones among them, best fit
        {"name": "path-ragged-best", "op": "path", "kind": "random", "traces": 301, "n": 701, "T": 1403,
         "ragged": True, "policy": "best"},
        # one very large model with weights-like tensors that outlive hundreds of ops
        {"name": "path-longtail", "op": "path", "kind": "longtail", "traces": 1, "n": 20000, "T": 10000,
         "ragged": False, "policy": "first"},
        # a serving fleet's sequence shapes planned together, best fit (the criterion of the paper's Sec. 2.3)
        {"name": "path-seq2seq-best", "op": "path", "kind": "seq2seq", "traces": 256, "n": 2000, "T": 4000,
         "ragged": False, "policy": "best"},
        # a plan refreshed for the same fleet where nothing else is wanted
        {"name": "plan-seq2seq", "op": "plan", "kind": "seq2seq", "traces": 64, "n": 1999, "T": 3999,
         "ragged": False, "policy": "first"},
        # memory curves of a corpus, for dashboards and lower bounds
        {"name": "profile-batch", "op": "profile", "kind": "random", "traces": 4096, "n": 512, "T": 1024,
         "ragged": False, "policy": "first"},
        # plans read back from a store checked before use, some of them stale
        {"name": "validate-batch", "op": "validate", "kind": "random", "traces": 4096, "n": 512, "T": 1024,
         "ragged": False, "policy": "first"},
        # the other strategy, for a comparison over the same fleet
        {"name": "breadth-seq2seq", "op": "breadth", "kind": "seq2seq", "traces": 256, "n": 2000, "T": 4000,
         "ragged": False, "policy": "first"},
        # how far the strategies are from the optimum, over a corpus of small graphs
        {"name": "optimal-tiny", "op": "optimal", "kind": "tiny", "traces": 4096, "n": 9, "T": 6, "ragged": False,
         "policy": "first"},
        # captured traces arrive in pinned host memory and the plans go back there
        {"name": "host-batch", "op": "host", "kind": "random", "traces": 4096, "n": 512, "T": 1024, "ragged": False,
         "policy": "first"},
    ]


def _spread(rng, lo, hi):
    """An integer of [lo, hi], evenly spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["path", "path", "path", "path", "plan", "profile", "validate", "breadth", "optimal", "host"])
    policy = rng.choice(["first", "best"])
    if op == "optimal":
        return {"op": op, "kind": "tiny", "traces": _spread(rng, 32, 4096), "n": rng.randint(4, 9), "T": 6,
                "ragged": bool(rng.getrandbits(1)), "policy": "first"}
    if op in ("path", "plan"):
        kind = rng.choice(["random", "random", "chain", "longtail", "seq2seq"])
    else:
        kind = rng.choice(["random", "random", "chain", "seq2seq"])
    ragged = kind == "random" and bool(rng.getrandbits(1))
    if kind == "random":
        n = _spread(rng, 16, 2000)
        traces = _spread(rng, 1, min(4096, (1 << 21) // n))
        T = max(8, int(n * rng.uniform(1.5, 3.0)))
    elif kind == "chain":
        T = _spread(rng, 40, 320)
        n = 2 * T + (T + 2) // 3
        traces = _spread(rng, 1, 64)
    elif kind == "longtail":
        n = _spread(rng, 1500, 20000)
        T = n // 2
        traces = 1 if n > 8000 else rng.randint(1, 3)
    else:
        n = _spread(rng, 300, 2000)
        T = 2 * n
        traces = _spread(rng, 1, 256)
    return {"op": op, "kind": kind, "traces": traces, "n": n, "T": T, "ragged": ragged, "policy": policy}


def _lifetimes(rng, alloc, T, p):
    return np.minimum(alloc + rng.geometric(p, size=alloc.shape), T)


def _log_uniform(rng, lo_e, hi_e, size):
    b = np.exp2(rng.uniform(lo_e, hi_e, size=size)).astype(np.int64)
    return (b + 63) // 64 * 64


def make_traces(case, seed):
    """The case's batch in host memory: structure of arrays with CSR offsets."""
    rng = np.random.default_rng([int(seed), case["traces"], case["n"], case["T"]])
    B, n, T = case["traces"], case["n"], case["T"]
    counts = np.full(B, n, dtype=np.int64)
    steps = np.full(B, T, dtype=np.int32)
    if case["ragged"]:
        # the case fixes the lengths (so that every seed has arrays of the same size), the seed their order
        counts = np.random.default_rng([B, n, T]).integers(1, n + 1, size=B).astype(np.int64)
        counts[0] = n
        rng.shuffle(counts)
        steps = np.maximum(8, counts * T // n).astype(np.int32)
    N = int(counts.sum())
    trace = np.repeat(np.arange(B), counts)
    Ti = steps[trace].astype(np.int64)
    kind = case["kind"]
    if kind == "tiny":
        alloc = rng.integers(0, T, size=N)
        free = np.minimum(alloc + rng.integers(1, T + 1, size=N), T)
        size = rng.integers(1, 4097, size=N)
    elif kind == "random":
        alloc = (rng.random(N) * Ti).astype(np.int64)
        free = _lifetimes(rng, alloc, Ti, 0.5)
        size = _log_uniform(rng, 6, 20, N)
    elif kind == "longtail":
        alloc = rng.integers(0, T, size=N)
        free = _lifetimes(rng, alloc, T, 0.4)
        size = _log_uniform(rng, 6, 26, N)
        for b in range(B):
            far = b * n + rng.permutation(n)[: n // 20]
            free[far] = np.minimum(alloc[far] + rng.integers(100, max(101, T // 2 + 1), size=far.size), T)
    elif kind == "seq2seq":
        alloc = rng.integers(0, T, size=N)
        free = _lifetimes(rng, alloc, T, 0.3)
        batch = np.repeat(rng.integers(1, 9, size=B), counts)
        length = np.repeat(rng.integers(1, 513, size=B), counts)
        hidden = np.where(rng.random(N) < 0.7, 1024, 4096)
        size = 4 * batch * hidden * np.where(rng.random(N) < 0.75, length, 1)
        for b in range(B):
            full = b * n + rng.permutation(n)[: n // 50]
            alloc[full] = 0
            free[full] = T
    else:  # chain: per op two activations, and a residual at every third
        op = np.concatenate([np.repeat(np.arange(T), 2), np.arange(0, T, 3)])
        first = np.concatenate([np.ones(2 * T, bool), np.zeros((T + 2) // 3, bool)])
        order = np.lexsort((~first, op))
        op, first = op[order], first[order]
        assert op.size == n
        alloc = np.tile(op, B)
        life = np.where(np.tile(first, B), rng.integers(1, 4, size=N), rng.integers(3, 5, size=N))
        free = np.minimum(alloc + life, T)
        per = -(-T // 5)  # five stages of consecutive ops
        shape = STAGES[rng.integers(0, 5, size=(B, 5))]
        bytes_ = 4 * shape[..., 0] * shape[..., 1] ** 2
        size = bytes_[trace, alloc // per]
    trace_ptr = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    profile_ptr = np.concatenate([[0], np.cumsum(steps, dtype=np.int64)]).astype(np.int64)
    return SimpleNamespace(trace_ptr=trace_ptr, steps=steps, profile_ptr=profile_ptr,
                           alloc_step=alloc.astype(np.int32), free_step=free.astype(np.int32),
                           size_bytes=size.astype(np.int64), n_traces=B, n_tensors=N, n_steps=int(profile_ptr[-1]),
                           max_tensors=int(counts.max()), max_steps=int(steps.max()))


def stored_offsets(ts, seed):
    """A plan read back from a store, made without the framework: every tensor
    above those allocated before it (always valid), in one trace of eight with
    one tensor moved to the bottom of the slab, as a stale plan has it."""
    rng = np.random.default_rng([int(seed), 77])
    trace = np.repeat(np.arange(ts.n_traces), np.diff(ts.trace_ptr))
    order = np.lexsort((ts.alloc_step, trace))
    before = np.cumsum(ts.size_bytes[order]) - ts.size_bytes[order]
    off = np.empty(ts.n_tensors, dtype=np.int64)
    off[order] = before
    counts = np.diff(ts.trace_ptr)
    base = np.where(counts > 0, np.concatenate([before, [0]])[np.minimum(ts.trace_ptr[:-1], ts.n_tensors)], 0)
    off -= base[trace]
    for b in range(0, ts.n_traces, 8):
        if counts[b] > 1:
            off[ts.trace_ptr[b] + rng.integers(counts[b])] = 0
    return off


def prepare(case, seed):
    ts = make_traces(case, seed)
    op = case["op"]
    st = SimpleNamespace(op=op, policy=case["policy"])
    if op == "host":
        st.path = mp.HostPath(ts, policy=case["policy"])
        return st
    st.batch = mp.DeviceBatch.from_host(ts, "cuda")
    dev = st.batch.device
    st.ws = mp.Workspace(dev)
    if op == "path":
        st.buffers = mp.PathBuffers(st.batch)
        return st
    st.status = torch.empty(ts.n_traces, dtype=torch.int32, device=dev)
    st.peak = torch.empty(ts.n_traces, dtype=torch.int64, device=dev)
    if op == "profile":
        st.profile = torch.empty(ts.n_steps, dtype=torch.int64, device=dev)
    elif op == "validate":
        st.offsets = torch.from_numpy(stored_offsets(ts, seed)).to(dev)
        st.verdict = torch.empty(ts.n_traces, dtype=torch.int32, device=dev)
        st.conflict = torch.empty(2 * ts.n_traces, dtype=torch.int32, device=dev)
        st.peak_status = torch.empty(ts.n_traces, dtype=torch.int32, device=dev)
    else:
        st.offsets = torch.empty(ts.n_tensors, dtype=torch.int64, device=dev)
    return st


def run(state):
    st, op = state, state.op
    if op == "host":
        return st.path.run()
    if op == "path":
        r = mp.plan_and_validate(st.batch, st.policy, st.buffers)
        return {"profile": r.profile, "peak_lb": r.peak_lb, "offsets": r.offsets, "plan_peak": r.plan_peak,
                "verdict": r.verdict, "conflict": r.conflict, "status": r.status}
    if op == "profile":
        profile, peak_lb, status = mp.live_profile(st.batch, st.profile, st.peak, st.status)
        return {"profile": profile, "peak_lb": peak_lb, "status": status}
    if op == "validate":
        verdict, conflict, status = mp.validate_plan(st.batch, st.offsets, st.verdict, st.conflict, st.status,
                                                     workspace=st.ws)
        plan_peak, _ = mp.peak(st.batch, st.offsets, st.peak, st.peak_status)
        return {"verdict": verdict, "conflict": conflict, "status": status, "plan_peak": plan_peak}
    if op == "plan":
        r = mp.plan_greedy_by_size(st.batch, st.policy, st.offsets, st.peak, st.status, workspace=st.ws)
    elif op == "breadth":
        r = mp.plan_greedy_by_breadth(st.batch, st.policy, st.offsets, st.peak, st.status, workspace=st.ws)
    else:
        r = mp.plan_optimal(st.batch, st.offsets, st.peak, st.status, workspace=st.ws)
    return {"offsets": r[0], "plan_peak": r[1], "status": r[2]}


def _sizes(case):
    """Expected tensors and steps of a batch (ragged traces average half the longest)."""
    share = 0.5 if case["ragged"] else 1.0
    return case["traces"] * case["n"] * share, case["traces"] * case["T"] * share


def work(case):
    N, S = _sizes(case)
    B, op = case["traces"], case["op"]
    read = 16 * N + 20 * B  # (alloc, free, size) per tensor; the CSR entries and step count per trace
    if op in ("path", "host"):
        moved = read + 8 * S + 8 * N + 32 * B
    elif op == "profile":
        moved = read + 8 * S + 12 * B
    elif op == "validate":
        moved = read + 8 * N + 24 * B
    else:
        moved = read + 8 * N + 12 * B
    return {"bytes": moved, "flops": 0}


def tolerance(case):
    return "exact"


# ---------------------------------------------------------------- plain restatement

def _profile(ts):
    trace = np.repeat(np.arange(ts.n_traces), np.diff(ts.trace_ptr))
    d = np.zeros(ts.n_steps + 1, dtype=np.int64)
    np.add.at(d, ts.profile_ptr[trace] + ts.alloc_step, ts.size_bytes)
    np.subtract.at(d, ts.profile_ptr[trace] + ts.free_step, ts.size_bytes)
    profile = np.cumsum(d)[:-1]  # a trace's differences sum to 0, so traces do not run into one another
    peak = np.array([profile[ts.profile_ptr[b]:ts.profile_ptr[b + 1]].max(initial=0) for b in range(ts.n_traces)],
                    dtype=np.int64)
    return profile, peak


def _greedy(a, f, s, order, policy):
    """Offsets of one trace, the tensors taken in the given order."""
    off = np.zeros(len(a), dtype=np.int64)
    done = np.zeros(len(a), dtype=bool)
    for i in order:
        j = np.flatnonzero(done & (a < f[i]) & (a[i] < f))
        if j.size:
            j = j[np.argsort(off[j], kind="stable")]
            top = np.maximum.accumulate(off[j] + s[j])
            floor = np.concatenate([[0], top[:-1]])
            gap = off[j] - floor
            fits = np.flatnonzero(gap >= s[i])
            if fits.size == 0:
                off[i] = top[-1]
            else:
                off[i] = floor[fits[0] if policy == "first" else fits[np.argmin(gap[fits])]]
        done[i] = True
    return off


def _order(case, a, f, s):
    if case["op"] != "breadth":
        return np.lexsort((np.arange(len(a)), a, -s))
    last = f - 1
    breadth = np.zeros(case["T"], dtype=np.int64)
    np.add.at(breadth, a, s)
    np.add.at(breadth, last, np.where(last != a, s, 0))
    later = breadth[last] > breadth[a]
    step = np.where(later, last, a)
    return np.lexsort((np.arange(len(a)), a, -s, step, -breadth[step]))


def exact(case, seed):
    op = case["op"]
    ts = make_traces(case, seed)
    B = ts.n_traces
    zeros = np.zeros(B, dtype=np.int32)
    a, f, s = ts.alloc_step.astype(np.int64), ts.free_step.astype(np.int64), ts.size_bytes
    part = [slice(int(ts.trace_ptr[b]), int(ts.trace_ptr[b + 1])) for b in range(B)]
    if op == "profile":
        profile, peak = _profile(ts)
        return {"profile": profile, "peak_lb": peak, "status": zeros}
    if op == "validate":
        off = stored_offsets(ts, seed)
        top = np.array([(off[q] + s[q]).max(initial=0) for q in part], dtype=np.int64)
        return {"verdict": None, "conflict": None, "status": zeros, "plan_peak": top}
    if op == "optimal":
        return None
    plan = None
    if ts.n_tensors <= 40000:  # a few seconds of plain numpy
        plan = np.concatenate([_greedy(a[q], f[q], s[q], _order(case, a[q], f[q], s[q]), case["policy"])
                               for q in part])
    top = None if plan is None else np.array([(plan[q] + s[q]).max(initial=0) for q in part], dtype=np.int64)
    if op in ("plan", "breadth"):
        return None if plan is None else {"offsets": plan, "plan_peak": top, "status": zeros}
    profile, peak = _profile(ts)
    return {"profile": profile, "peak_lb": peak, "offsets": plan, "plan_peak": top,
            "verdict": np.ones(B, dtype=np.int32),
            "conflict": np.full(2 * B if op == "host" else (B, 2), -1, dtype=np.int32), "status": zeros}
