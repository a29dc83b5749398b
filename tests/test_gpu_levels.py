"""The levelled composer at the edges of its plan, against the oracle: chains of 1 to 130 ops (segments hold at most 64,
warps take 4 and 8 rows at a time), joins of 1 to 150 inputs (4 in the head program, 6 in the first piece of a list, 8 in
each further one; more than 128 segments a level take two steps), asynchronous collectives that make overlap candidates of
the chains beside them, and full and partial scenario blocks of every width."""

import numpy as np
import pytest

import oracle
from paper_2412_12487_gb300 import Echo
from paper_2412_12487_gb300 import workloads as W

from . import smallgraphs as SG
from .test_gpu_parity import assert_same, run_gpu

pytestmark = pytest.mark.gpu


def _joins(ranks, lengths):
    """Rounds of a chain on every rank and a join of all ranks; on stream 2 a collective of the round that only the last
    op waits for."""
    ops, queues, waits = [], {(r, k): [] for r in range(ranks) for k in range(3)}, []
    everyone = list(range(ranks))
    join = None
    for i in range(len(lengths)):
        tails = []
        for r in everyone:
            for n in range(lengths[(i + r) % len(lengths)]):
                queues[(r, 0)].append(len(ops))
                ops.append({"kind": W.KIND_COMPUTE, "kclass": r % 3, "preds": [join] if n == 0 and join is not None else []})
            tails.append(len(ops) - 1)
        for stream in (1, 2):
            for r in everyone:
                queues[(r, stream)].append(len(ops))
            if stream == 1:
                join = len(ops)
            else:
                waits.append(len(ops))
            ops.append({"kind": W.KIND_COLL, "group": 0, "cc_type": W.CC_ALLREDUCE, "cc_algo": W.ALGO_AUTO,
                        "cc_bytes": 1 << (10 + i), "preds": tails})
    queues[(0, 0)].append(len(ops))
    ops.append({"kind": W.KIND_COMPUTE, "kclass": 0, "preds": waits + [join]})
    return SG.graph_from_lists(ranks, 3, ops, queues, [everyone], gpus_per_node=4)


@pytest.mark.parametrize("sigma", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("ranks", [1, 4, 5, 10, 11, 19, 150])
def test_chain_and_join_edges_bit_exact(sigma, ranks, monkeypatch):
    monkeypatch.setenv("ECHO_COMPOSE_KERNEL", "pipelined")
    monkeypatch.setenv("ECHO_SIGMA", str(sigma))
    g = _joins(ranks, [1, 3, 4, 5, 7, 8, 9] + ([63, 64, 65, 130] if ranks < 100 else [12]))
    rng = np.random.default_rng(100 * sigma + ranks)
    with Echo(0) as e:
        e.set_profiling(True)
        for S in (sigma, 2 * sigma + 1):
            sc = SG.random_scenarios(rng, g, S, max_dur=20_000)
            for refine, model, interval in ((0, 0, 0), (1, 0, 0), (2, 1, 1)):
                got = run_gpu(g, sc, refine, ctx=e, overlap_model=model, comm_interval=interval)
                assert got["info"]["sigma"] == sigma
                # (a plan that does not fit takes the staged composer, which has a name of its own)
                assert {k for k in e.read_profile() if k.startswith("compose")} == {"compose"} | ({"compose_adjusted"} if refine else set())
                want = oracle.compose(g, sc, refine_passes=refine, overlap_model=model, comm_interval=interval)
                assert_same(got, want, g, refine)


@pytest.mark.parametrize("sigma", [1, 2, 4, 8, 16])
def test_debug_bounds_of_every_block_width(sigma, monkeypatch):
    """The checking variant of every role (sums in place and stores by rows for blocks of 1 and 2, walks above; lists of
    inputs; candidates): no check fails on well-formed graphs, and the times are the oracle's."""
    monkeypatch.setenv("ECHO_COMPOSE_KERNEL", "pipelined")
    monkeypatch.setenv("ECHO_SIGMA", str(sigma))
    rng = np.random.default_rng(300 + sigma)
    graphs = [_joins(11, [1, 3, 64, 65]), _joins(150, [1, 9, 12])]
    graphs += [SG.random_graph(rng, int(rng.integers(20, 300)), max_ranks=5, max_streams=8, p_edge=0.03) for _ in range(4)]
    with Echo(0) as e:
        e.set_profiling(True)
        for g in graphs:
            sc = SG.random_scenarios(rng, g, sigma + 1, max_dur=20_000)
            for refine, model, interval in ((0, 0, 0), (2, 1, 1)):
                e.load_graph(g)
                e.load_scenarios(sc)
                e.estimate_collectives()
                e.compose(refine_passes=refine, overlap_model=model, comm_interval=interval, debug_bounds=True)
                assert "compose" in e.read_profile()
                st, fn = e.read_times()
                got = dict(start=st, finish=fn, makespan=e.read_makespan(), cc=e.read_cc(), ov=e.read_overlap())
                assert_same(got, oracle.compose(g, sc, refine_passes=refine, overlap_model=model, comm_interval=interval), g, refine)


@pytest.mark.parametrize("ranks,S,kernel", [(1000, 70, None), (1000, 17, "pipelined"), (1000, 17, "staged"), (40, 5, "staged")])
def test_without_a_levelled_plan(ranks, S, kernel, monkeypatch):
    """More live tails than half of a block's shared memory holds (1000 in blocks of 16): the staged composer runs, and
    reads the validator's durations where they are, without a full matrix made of them."""
    monkeypatch.setenv("ECHO_SIGMA", "16" if ranks == 1000 else "1")
    if kernel:
        monkeypatch.setenv("ECHO_COMPOSE_KERNEL", kernel)
    g = _joins(ranks, [1, 2, 5, 65] if ranks == 40 else [1, 2, 5])
    sc = SG.random_scenarios(np.random.default_rng(S), g, S, max_dur=20_000)
    with Echo(0) as e:
        e.set_profiling(True)
        for refine, model, interval in ((0, 0, 0), (1, 0, 0), (2, 1, 1), (3, 0, 0)):
            for debug in (False, True):
                e.load_graph(g)
                e.load_scenarios(sc)
                e.estimate_collectives()
                e.compose(refine_passes=refine, overlap_model=model, comm_interval=interval, debug_bounds=debug)
                st, fn = e.read_times()
                got = dict(start=st, finish=fn, makespan=e.read_makespan(), cc=e.read_cc(), ov=e.read_overlap())
                want = oracle.compose(g, sc, refine_passes=refine, overlap_model=model, comm_interval=interval)
                assert_same(got, want, g, refine)
                ran = e.read_profile()
                assert ran["compose_staged"][0] == refine + 1
                assert not {"scatter_candidates", "compose", "compose_adjusted", "compose_direct"} & set(ran)


@pytest.mark.parametrize("lengths,S,sigma,ran", [([30], 1217, 8, "compose"), ([1, 2, 5], 1217, 16, "compose_staged"),
                                                 ([30], 5, 32, "compose"), ([1, 2, 5], 5, 1, "compose"),
                                                 ([30], 200, 2, "compose")])
def test_choice_among_composers_that_exist(lengths, S, sigma, ran):
    """950 ranks: 1217 scenarios ask for blocks of 16, in which the tails do not fit.  Long chains take the levelled
    composer in blocks of 8, short ones the staged one; few scenarios the dataflow composer where a rank's chain is long
    beside its joins; narrower blocks have a levelled plan of their own."""
    g = _joins(950, lengths)
    sc = SG.random_scenarios(np.random.default_rng(S), g, S, max_dur=20_000)
    with Echo(0) as e:
        e.set_profiling(True)
        e.load_graph(g)
        for _ in range(2):  # (a second batch keeps the first one's choice)
            e.load_scenarios(sc)
            e.estimate_collectives()
            e.read_profile()
            e.compose()
            st, fn = e.read_times()
            got = dict(start=st, finish=fn, makespan=e.read_makespan(), cc=e.read_cc(), ov=e.read_overlap())
            assert e.info()["sigma"] == sigma
            assert [k for k in e.read_profile() if k.startswith("compose")][0] == ran
            assert_same(got, oracle.compose(g, sc, threads=8), g)


@pytest.mark.parametrize("kernel", ["dataflow", "staged", "direct", "levelled"])
def test_contexts_with_different_shared_memory(kernel, monkeypatch):
    """Blocks of two contexts need different amounts of shared memory; neither's batches lower the other's limit."""
    monkeypatch.setenv("ECHO_COMPOSE_KERNEL", kernel)
    shapes = [W.GPTConfig("case", layers=4, hidden=1024, heads=8, seq=512, tp=tp, pp=2, dp=2, microbatches=4, virtual_stages=v, n_scen=7)
              for tp, v in ((8, 2), (2, 1))]  # blocks of 8 ranks with 8 timelines; of 2 with fewer
    batches = []
    for c in shapes:
        g = W.build_gpt_graph(c)
        sc = W.make_scenarios(g, c, n_scen=7)
        batches.append((g, sc, oracle.compose(g, sc)))
    contexts = [Echo(0) for _ in batches]
    try:
        for e, (g, sc, _) in zip(contexts, batches):
            e.load_graph(g)
            e.load_scenarios(sc)
        for order in ((0, 1), (1, 0), (0, 1)):
            for i in order:
                contexts[i].load_scenarios(batches[i][1])
            for i in order:
                contexts[i].estimate_collectives()
                contexts[i].compose()
                assert np.array_equal(contexts[i].read_times()[1], batches[i][2].finish)
    finally:
        for e in contexts:
            e.close()
