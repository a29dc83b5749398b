"""Reading times back from scenario blocks of every width: the tiled paths (32 scenarios and more, columns of 192 and more)
and the other one, op and scenario ranges that start and end inside tiles, host and device buffers; and the load's tiles
and sums (32 and 64 bits), through the times they give."""
import numpy as np
import pytest

import oracle
from paper_2412_12487_gb300 import Echo, EchoError
from paper_2412_12487_gb300 import workloads as W
from tests import smallgraphs as SG

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", ["1", "2", "16", None])
@pytest.mark.parametrize("S", [1, 33, 97, 401])
def test_ranges_host_and_device(sigma, S, monkeypatch):
    import torch

    if sigma is not None:
        monkeypatch.setenv("ECHO_SIGMA", sigma)
    c = W.GPTConfig(**{**W.config("tiny").__dict__, "fixed_scenario": False})
    g = W.build_gpt_graph(c)
    sc = W.make_scenarios(g, c, n_scen=S)
    want = oracle.compose(g, sc)
    V = g.n_ops
    with Echo(0) as e:
        e.load_graph(g)
        for bits in (64, 32):
            e.load_scenarios(sc, dur=sc.dur.astype(np.int32) if bits == 32 else None)
            e.estimate_collectives()
            e.compose()
            for op0, op1 in ((0, V), (0, 1), (31, 33), (V - 65, V)):
                for s0, s1 in ((0, S), (S // 2, S), (0, max(1, S - 1)), (S - 1, S)):
                    st, fn = e.read_times(op0, op1, s0=s0, s1=s1)
                    assert np.array_equal(st, want.start[op0:op1, s0:s1])
                    assert np.array_equal(fn, want.finish[op0:op1, s0:s1])
                    ds = torch.full((op1 - op0, s1 - s0), -1, dtype=torch.int64, device="cuda")
                    df = torch.full_like(ds, -1)
                    for a, b in ((ds, df), (None, df), (ds, None)):
                        rc = e.lib.echo_read_times(e.h, op0, op1, s0, s1, a.data_ptr() if a is not None else None,
                                                   b.data_ptr() if b is not None else None)
                        assert rc == 0
                    assert np.array_equal(ds.cpu().numpy(), want.start[op0:op1, s0:s1])
                    assert np.array_equal(df.cpu().numpy(), want.finish[op0:op1, s0:s1])
        dm = torch.full((S,), -1, dtype=torch.int64, device="cuda")
        assert e.lib.echo_read_makespan(e.h, dm.data_ptr()) == 0
        assert np.array_equal(dm.cpu().numpy(), want.makespan) and np.array_equal(e.read_makespan(), want.makespan)
        bad = sc.dur.copy()
        bad[np.nonzero(g.kind == W.KIND_COMPUTE)[0][-1], S - 1] = -1
        with pytest.raises(EchoError) as ei:
            e.load_scenarios(sc, dur=bad)
        assert ei.value.code == 1


def test_sums_still_refuse_what_could_overflow():
    # durations whose sum passes 2^62 in one scenario only, with halves that carry into each other
    c = W.config("tiny")
    g = W.build_gpt_graph(c)
    sc = W.make_scenarios(g, c, n_scen=3)
    local = np.nonzero(g.kind == W.KIND_COMPUTE)[0]
    for each, refused in (((1 << 62) // len(local) + (1 << 33), True), ((1 << 56) // len(local) + 12345, False)):
        sc.dur[local, 1] = each
        with Echo(0) as e:
            e.load_graph(g)
            e.load_scenarios(sc)
            if refused:
                with pytest.raises(EchoError) as ei:
                    e.estimate_collectives()
                assert ei.value.code == 8
            else:
                e.estimate_collectives()
                e.compose()
                assert np.array_equal(e.read_makespan(), oracle.compose(g, sc).makespan)


@pytest.mark.parametrize("S", [32 * 65535, 32 * 65535 + 1])
def test_more_scenarios_than_the_tiles_have_columns(S):
    g = SG.graph_from_lists(1, 2, [{"kind": W.KIND_COMPUTE, "kclass": 0, "preds": []} for _ in range(3)], {(0, 0): [0, 1, 2]}, [[0]],
                            gpus_per_node=1)
    sc = SG.random_scenarios(np.random.default_rng(1), g, S, max_dur=1000)
    want = np.cumsum(sc.dur, axis=0)
    with Echo(0) as e:
        e.load_graph(g)
        e.load_scenarios(sc)
        e.estimate_collectives()
        e.compose(refine_passes=0)
        for op0, op1 in ((0, 2), (0, 3)):  # tiles in the caller's order; every op, S past the end of the tiles' columns
            st, fn = e.read_times(op0, op1)
            assert np.array_equal(fn, want[op0:op1]) and np.array_equal(st, (want - sc.dur)[op0:op1])
        assert np.array_equal(e.read_makespan(), want[-1])
