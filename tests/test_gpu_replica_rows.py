"""The comparison of replica rows finds one differing duration wherever it is: rows compared in 16-byte words and in the
durations' own, of fewer words than a team's lanes take at once, of exactly as many, and of more."""
import dataclasses

import numpy as np
import pytest

from paper_2412_12487_gb300 import Echo
from paper_2412_12487_gb300 import workloads as W
from tests.test_replicas import originals

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 127, 128, 129, 256, 516, 1030])
def test_one_difference_anywhere(S):
    c = dataclasses.replace(W.config("tiny"), identical_replicas=True, fixed_scenario=False)
    g = W.build_gpt_graph(c)
    sc = W.make_scenarios(g, c, n_scen=S)
    dup = np.nonzero((originals(g) != np.arange(g.n_ops)) & (g.kind == W.KIND_COMPUTE))[0]
    with Echo(0) as e:
        e.load_graph(g)
        for dt in (np.int64, np.int32):
            dur = sc.dur.astype(dt)
            for op, s in [(None, 0)] + [(x, s) for x in (dup[0], dup[-1]) for s in sorted({0, S // 2, S - 1})]:
                if op is not None:
                    dur[op, s] += 1
                e.load_scenarios(sc, dur=dur)
                assert e.info()["replicas_folded"] == (1 if op is None else 0), (op, s)
                if op is not None:
                    dur[op, s] -= 1
