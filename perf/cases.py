"""The work that a user of this library has it do, as cases to measure.

Four kinds of pass, each through the public entry points:

* ``sweep``: the scenarios are loaded; one pass estimates the collectives, composes and reads the result (a user
  comparing options on one batch).
* ``batch``: a new scenario batch from host memory, then the same (a what-if loop: every pass uploads its durations).
* ``query``: standalone collective-cost queries from host arrays (``Echo.cc_query``).
* ``query_device``: the same with arrays that live on the device (``echo_cc_query_noalloc``).

A timeline case gives its workload's shape in the terms of ``workloads.GPTConfig`` and what is read back:
``makespan`` (the step times), ``times`` (start and finish of every op into host arrays), ``times_device`` (the same
into device buffers) or ``overlap`` (the validator's decisions, with the step times).  Times are integers, so their
tolerance is "exact"; the queries are fp64.
"""
import ctypes
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_2412_12487_gb300 import Echo
from paper_2412_12487_gb300 import echo as E
from paper_2412_12487_gb300 import workloads as W

SHAPE = ("layers", "hidden", "heads", "seq", "tp", "pp", "dp", "microbatches", "virtual_stages", "identical_replicas")


def _timeline(name, config, scenarios, kind="sweep", bits=64, read="makespan", refine=1, model=0, interval=0, policy=0,
              replicas=False):
    c = W.config(config)
    case = {"name": name, "kind": kind, "scenarios": scenarios, "bits": bits, "read": read, "refine": refine,
            "model": model, "interval": interval, "policy": policy}
    case.update({k: getattr(c, k) for k in SHAPE})
    case["identical_replicas"] = replicas
    return case


def listed():
    return [
        # one step of the smallest workload, from its durations to its timeline: an interactive what-if, where
        # launches and synchronisations are all there is
        _timeline("tiny-1-batch-times", "tiny", 1, kind="batch", read="times"),
        # one scenario of the 64-rank workload and its whole timeline (what a trace viewer shows)
        _timeline("gpt1.3b-1-times", "gpt1.3b", 1, read="times"),
        # the 64-rank workload at its own batch width: step times of loaded scenarios
        _timeline("gpt1.3b-256", "gpt1.3b", 256),
        # the same as a what-if loop runs it: every pass brings new 64-bit durations
        _timeline("gpt1.3b-256-batch", "gpt1.3b", 256, kind="batch"),
        # the validator's variants on a ragged batch: intervals from each rank's launch, proportional slowdown, two
        # validator passes, another all-reduce policy; its decisions are read back
        _timeline("gpt1.3b-45-variants", "gpt1.3b", 45, read="overlap", refine=2, model=1, interval=1, policy=3),
        # identical data-parallel replicas, folded, with a new batch in 32 bits each pass
        _timeline("gpt1.3b-500-folded-batch", "gpt1.3b", 500, kind="batch", bits=32, replicas=True),
        # the 96-rank workload at its own batch width: the headline
        _timeline("gpt175b-1024", "gpt175b", 1024, bits=32),
        # a ragged batch of it, with every op's times left on the device for further analysis
        _timeline("gpt175b-250-times", "gpt175b", 250, read="times_device"),
        # 1024 ranks, interleaved schedule, 8 timelines a rank, few scenarios
        _timeline("gpt175b-1024ranks-64", "gpt175b-1024-small", 64),
        # collective-cost queries: the estimator sweep on device arrays, and a tool's table from host arrays
        {"name": "query-1M-device", "kind": "query_device", "n": 1_000_000},
        {"name": "query-20k-host", "kind": "query", "n": 20_011},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.2:
        return {"kind": rng.choice(["query", "query_device"]), "n": _log_int(rng, 1000, 1_000_000)}
    while True:
        tp, pp, dp = rng.choice([1, 2, 4, 8]), rng.choice([1, 2, 3, 4, 6, 8]), rng.choice([1, 2, 3, 4, 8])
        virtual = rng.choice([1, 1, 2]) if pp > 1 else 1
        layers = pp * virtual * rng.randint(1, 4)
        heads = rng.choice([16, 32, 96])
        micro = pp * rng.randint(1, 4)
        local = layers * micro * 46 * tp * dp  # compute ops, about
        scen = _log_int(rng, 1, 1024)
        if 800 <= local <= 250_000 and local * scen <= 200_000_000:
            break
    kind = rng.choice(["sweep", "sweep", "batch"])
    read = rng.choice(["makespan", "makespan", "times_device"] + (["times", "overlap"] if local * scen < 2_000_000 else []))
    return {"kind": kind, "scenarios": scen, "bits": rng.choice([32, 64]), "read": read, "refine": rng.choice([0, 1, 1, 1, 2, 3]),
            "model": rng.choice([0, 0, 1]), "interval": rng.choice([0, 0, 1]), "policy": rng.choice([0, 0, 0, 1, 2, 3]),
            "layers": layers, "hidden": 128 * heads, "heads": heads, "seq": rng.choice([512, 2048, 4096]), "tp": tp, "pp": pp,
            "dp": dp, "microbatches": micro, "virtual_stages": virtual,
            # (replicas have the same group shapes only where each fills whole nodes of 8)
            "identical_replicas": bool(dp > 1 and tp * pp % 8 == 0 and rng.random() < 0.6)}


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=4)
def _graph(key):
    """The execution graph of a shape, and which ops share a noise draw (identical replicas do)."""
    shape = dict(key)
    g = W.build_gpt_graph(W.GPTConfig("case", n_scen=1, **shape))
    share = np.unique(g.noise, return_inverse=True)[1] if shape["identical_replicas"] else None
    return g, share


def _inputs(case, seed):
    """Graph, scenario parameters and durations of a timeline case, all drawn from the seed as the workload generator
    draws them; durations in pinned host memory, as a loop that uploads them keeps them."""
    g, share = _graph(tuple((k, case[k]) for k in SHAPE))
    rng = np.random.Generator(np.random.PCG64(seed))
    noise = np.exp(rng.normal(0.0, 0.1, size=g.n_ops if share is None else int(share.max()) + 1))
    g = dataclasses.replace(g, noise=noise if share is None else noise[share])
    S = case["scenarios"]
    sc = W.scenario_params(W.GPTConfig("case", n_scen=S, scen_seed=seed, **{k: case[k] for k in SHAPE}), S)
    dtype = torch.int32 if case["bits"] == 32 else torch.int64
    dur = torch.empty((g.n_ops, S), dtype=dtype, pin_memory=True)
    local = (g.kind == W.KIND_COMPUTE) | (g.kind == W.KIND_MEMCPY)
    work = torch.from_numpy(np.where(local, g.work * g.noise, 0.0)).cuda()
    peak = torch.from_numpy(sc.peak_flop_per_ns).cuda()
    rows = max(1, (1 << 25) // S)
    for i in range(0, g.n_ops, rows):
        dur[i:i + rows].copy_((work[i:i + rows, None] / peak[None, :]).round_().to(dtype))
    return g, sc, dur


def prepare(case, seed):
    if case["kind"].startswith("query"):
        q = W.make_cc_queries(case["n"], seed=seed)
        if case["kind"] == "query":
            return {"case": case, "echo": Echo(0), "queries": q}
        arrays = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (
            q.cc_type, q.cc_algo, q.nbytes, q.n_ranks, q.n_nodes, q.alpha_ns, q.bw_intra, q.lat_intra, q.bw_inter,
            q.lat_inter, q.delta)]
        out = torch.empty(q.n, dtype=torch.float64, device="cuda")
        desc = E.CCQueryDesc(q.n, *[x.data_ptr() for x in arrays], 0, None, None)
        return {"case": case, "lib": E.load_library(), "arrays": arrays, "desc": desc, "out": out}
    g, sc, dur = _inputs(case, seed)
    e = Echo(0)
    e.load_graph(g)
    state = {"case": case, "echo": e}
    if case["kind"] == "batch":
        state.update(sc=sc, dur=dur)
    else:
        e.load_scenarios(sc, dur=dur)
    if case["read"] == "times_device":
        state["times"] = [torch.empty((g.n_ops, case["scenarios"]), dtype=torch.int64, device="cuda") for _ in range(2)]
    return state


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    if case["kind"] == "query":
        return state["echo"].cc_query(state["queries"])
    if case["kind"] == "query_device":
        rc = state["lib"].echo_cc_query_noalloc(ctypes.byref(state["desc"]), state["out"].data_ptr(),
                                                torch.cuda.current_stream().cuda_stream)
        if rc:
            raise RuntimeError(E.STATUS_NAMES[rc])
        return state["out"]
    e = state["echo"]
    if case["kind"] == "batch":
        e.load_scenarios(state["sc"], dur=state["dur"])
    e.estimate_collectives()
    e.compose(refine_passes=case["refine"], overlap_model=case["model"], comm_interval=case["interval"],
              ar_algo_policy=case["policy"])
    out = {"makespan": e.read_makespan()}
    if case["read"] == "times":
        out["start"], out["finish"] = e.read_times()
    elif case["read"] == "times_device":  # the C call with device buffers (the binding's own arrays are host arrays)
        start, finish = state["times"]
        rc = e.lib.echo_read_times(e.h, 0, start.shape[0], 0, start.shape[1], start.data_ptr(), finish.data_ptr())
        if rc:
            raise RuntimeError(E.STATUS_NAMES[rc])
        out["start"], out["finish"] = start, finish
    elif case["read"] == "overlap":
        out["overlap"] = e.read_overlap()
    return out


def work(case):
    if case["kind"].startswith("query"):
        # the arrays in (2 bytes, a size, two counts, six fp64 parameters) and one fp64 out; two chunk divides, two
        # transfer divides and about a dozen multiplies and adds a query
        return {"bytes": 74 * case["n"], "flops": 16 * case["n"]}
    g, _ = _graph(tuple((k, case[k]) for k in SHAPE))
    V, S = g.n_ops, case["scenarios"]
    if case["identical_replicas"]:  # one copy is composed; a batch's rows are all read
        V //= case["dp"]
    local = int(V * np.mean((g.kind == W.KIND_COMPUTE) | (g.kind == W.KIND_MEMCPY)))
    n = local * S * case["bits"] // 8 + 8 * V * S  # durations in, finish times out
    if case["kind"] == "batch":
        n += g.n_ops * S * case["bits"] // 8
    if case["read"].startswith("times"):
        n += 16 * g.n_ops * S
    elif case["read"] == "overlap":
        n += g.n_ops * S
    # one addition and about two maxima per op, scenario and composition
    return {"bytes": n + 8 * S, "flops": 3 * V * S * (1 + case["refine"])}


def tolerance(case):
    # The times are whole nanoseconds with one right value each.  A query is a chain of about a dozen fp64 operations on
    # positive terms: with its sums and products in another order (the plain form below, rewritten) 1M queries moved by
    # 1.1e-16 (2-norm) and 4.4e-16 (largest); four times that is allowed.
    return {"rel": 5e-16, "max": 2e-15} if case["kind"].startswith("query") else "exact"


# ---------------------------------------------------------------------------------------
# the same in plain numpy
# ---------------------------------------------------------------------------------------
_CHUNKS = ((4 << 20, 18000), (8 << 20, 36000), (64 << 20, 72000), (128 << 20, 144000), (1 << 62, 288000))


def _cost(typ, algo, size, N, M, K, alpha, Ba, La, Be, Le, delta):
    """Time of collectives; every argument an array (they broadcast)."""
    typ, algo, size, N, M, K = np.broadcast_arrays(typ, algo, size, N, M, K)
    chunk = np.select([size <= m for m, _ in _CHUNKS], [c for _, c in _CHUNKS])
    L, B = np.where(M > 1, Le, La), np.where(M > 1, Be, Ba)
    one = np.maximum(1, -(-size // chunk))
    sendrecv = alpha + one * (L + size / one / B)
    eta = np.maximum(1, -(-size // (N * chunk)))
    ring = alpha + np.where(typ == 0, 2, 1) * eta * (N - 1) * (L + size / (N.astype(float) * eta) / B)
    ring = ring + np.where(typ == 1, 0.0, delta * size)
    part = size / one
    beta = La + part / Ba
    gamma = np.where(M > 1, Le + part / Be, beta)
    tree = alpha + gamma * (one - 1) + 2.0 * beta * (K - 1) + 2.0 * gamma * np.log2(M) + delta * size
    t = np.where(typ == 3, sendrecv, ring)
    t = np.where((typ == 0) & (algo == 1), tree, t)
    t = np.where((typ == 0) & (algo == 2), np.minimum(ring, tree), t)
    return np.where((N <= 1) | (size <= 0), 0.0, t)


def _covered(intervals, x):
    """How much of (-inf, x] the union of the (start, end) rows covers."""
    a = intervals[np.argsort(intervals[:, 0], kind="stable")]
    end = np.maximum.accumulate(a[:, 1])
    new = np.r_[True, a[1:, 0] > end[:-1]]
    lo = a[new, 0]
    hi = end[np.r_[np.nonzero(new)[0][1:] - 1, len(a) - 1]]
    done = np.r_[0, np.cumsum(hi - lo)]
    i = np.searchsorted(lo, x, side="right") - 1
    return np.where(i < 0, 0, done[i] + np.minimum(x, hi[i]) - lo[i])


def exact(case, seed):
    if case["kind"].startswith("query"):
        q = W.make_cc_queries(case["n"], seed=seed)
        N, M = q.n_ranks.astype(np.int64), q.n_nodes.astype(np.int64)
        return _cost(q.cc_type, q.cc_algo, q.nbytes, N, M, -(-N // M), q.alpha_ns, q.bw_intra, q.lat_intra, q.bw_inter,
                     q.lat_inter, q.delta)
    S = case["scenarios"]
    g, _ = _graph(tuple((k, case[k]) for k in SHAPE))
    if g.n_ops > 160_000 or g.n_ops * S > 8_000_000:  # over about 20 seconds
        return None
    g, sc, dur = _inputs(case, seed)
    V, R, NS = g.n_ops, g.n_ranks, g.n_streams
    d = dur.numpy().astype(np.int64)
    comm = g.kind >= W.KIND_COLL
    cost = {}
    for v in np.nonzero(comm)[0]:
        ranks = g.grp_rank[g.grp_off[g.group[v]]:g.grp_off[g.group[v] + 1]]
        n = len(ranks)
        per = np.unique(ranks // g.gpus_per_node, return_counts=True)[1]
        algo = int(g.cc_algo[v]) if case["policy"] == 0 else case["policy"] - 1
        key = (int(g.cc_type[v]), algo, int(g.cc_bytes[v]), n, len(per), int(per.max()))
        if key not in cost:
            cost[key] = np.rint(_cost(*[np.int64(k) for k in key], sc.alpha_ns, sc.bw_intra, sc.lat_intra, sc.bw_inter,
                                      sc.lat_inter, sc.delta)).astype(np.int64)
        d[v] = cost[key]
    before = [list(g.pred_idx[g.pred_off[v]:g.pred_off[v + 1]]) for v in range(V)]
    queues = [[g.q_ops[g.q_off[r * NS + k]:g.q_off[r * NS + k + 1]] for k in range(NS)] for r in range(R)]
    for q in (q for rank in queues for q in rank):
        for u, v in zip(q[:-1], q[1:]):
            before[v].append(u)
    after, open_ = [[] for _ in range(V)], np.array([len(b) for b in before])
    for v, b in enumerate(before):
        for u in b:
            after[u].append(v)
    order = list(np.nonzero(open_ == 0)[0])
    for u in order:
        for v in after[u]:
            open_[v] -= 1
            if not open_[v]:
                order.append(v)

    def compose(dur_now):
        f = np.zeros((V, S), np.int64)
        for v in order:
            f[v] = dur_now[v] + (f[before[v]].max(axis=0) if before[v] else 0)
        return f

    now, slowed = d, np.zeros((V, S), np.uint8)
    f = compose(now)
    for _ in range(case["refine"]):
        after_pass, slowed = d.copy(), np.zeros((V, S), np.uint8)
        start = f - now
        for r in range(R):
            mine = queues[r][0]
            here = set(int(v) for q in queues[r] for v in q)
            lo, hi = [], []
            for q in queues[r][1:]:
                for i, w in enumerate(q):
                    if not comm[w]:
                        continue
                    if case["interval"]:
                        mine_before = [q[i - 1]] * (i > 0) + [u for u in g.pred_idx[g.pred_off[w]:g.pred_off[w + 1]] if int(u) in here]
                        lo.append(f[mine_before].max(axis=0) if mine_before else np.zeros(S, np.int64))
                    else:
                        lo.append(start[w])
                    hi.append(f[w])
            if not lo or not len(mine):
                continue
            lo, hi = np.array(lo), np.array(hi)
            length = np.empty((len(mine), S), np.int64)
            for s in range(S):
                rows = np.stack([lo[:, s], hi[:, s]], axis=1)
                rows = rows[rows[:, 1] > rows[:, 0]]
                length[:, s] = _covered(rows, f[mine, s]) - _covered(rows, start[mine, s]) if len(rows) else 0
            factor = sc.slowdown[g.kclass[mine]]
            long = d[mine] + (factor - 1.0) * length if case["model"] else d[mine] * factor
            hit = (length > 0) & (now[mine] > 0)
            after_pass[mine] = np.where(hit, np.rint(long).astype(np.int64), d[mine])
            slowed[mine] = hit
        now = after_pass
        f = compose(now)
    out = {"makespan": f.max(axis=0)}
    if case["read"].startswith("times"):
        out["start"], out["finish"] = f - now, f
    elif case["read"] == "overlap":
        out["overlap"] = slowed
    return out
