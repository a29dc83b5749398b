"""Collective-time queries: counts around a block's, mixed forms and one form only, byte counts at the edges of the
integer shortcuts (2^20 chunk rounds, 2^31 and 2^53 as a product, 2^40 as a chunk), and an output that is an input.
Every estimate is the same single operations in the same order as the oracle's, so the two are equal to the last bit."""
import ctypes as C

import numpy as np
import pytest

import oracle
from paper_2412_12487_gb300 import echo as E
from paper_2412_12487_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TABLES = [None, ([1 << 62], [1]), ([1 << 30, 1 << 62], [3, 1 << 41])]


def _queries(rng, n, forms):
    q = W.make_cc_queries(n, seed=int(rng.integers(1 << 30)))
    t, a = [np.array(x, np.uint8) for x in zip(*forms)]
    pick = rng.integers(0, len(forms), size=n)
    q.cc_type, q.cc_algo = t[pick], a[pick]
    edge = np.array([0, 1, 2, 3, 2 ** 20, 2 ** 31, 2 ** 40, 2 ** 53, 2 ** 58])
    q.nbytes = np.where(rng.random(n) < 0.5, np.maximum(edge[rng.integers(0, len(edge), size=n)] + rng.integers(-1, 2, size=n), 0),
                        q.nbytes).astype(np.int64)
    q.n_ranks = np.where(rng.random(n) < 0.1, 1, q.n_ranks).astype(np.int32)
    q.n_nodes = np.where(q.n_ranks == 1, 1, q.n_nodes).astype(np.int32)
    q.n_nodes = np.minimum(q.n_nodes, q.n_ranks)
    if n > 4000:  # more nodes than the table of logarithms holds
        q.n_ranks[7], q.n_nodes[7] = 300_000, 5000
    return q


def _want(q, table):
    lib = oracle._load()
    prm = np.ascontiguousarray(np.stack([q.alpha_ns, q.bw_intra, q.lat_intra, q.bw_inter, q.lat_inter, q.delta], 1))
    tab = [np.array(x, np.int64) for x in table] if table else None
    args = (len(tab[0]), C.c_void_p(tab[0].ctypes.data), C.c_void_p(tab[1].ctypes.data)) if tab else (0, None, None)
    out = np.empty(q.n)
    for i in range(q.n):
        N, M = int(q.n_ranks[i]), int(q.n_nodes[i])
        out[i] = lib.oracle_cc_ns(int(q.cc_type[i]), int(q.cc_algo[i]), int(q.nbytes[i]), N, M, -(-N // M),
                                  float(np.log2(np.float64(M))), C.c_void_p(prm.ctypes.data + 48 * i), *args)
    return out


FORMS = {"mixed": [(0, 0), (0, 1), (0, 2), (1, 0), (2, 0), (3, 0)], "trees": [(0, 1), (0, 2)], "linear": [(0, 0), (1, 0), (2, 0), (3, 0)]}


@pytest.mark.parametrize("forms", list(FORMS))
@pytest.mark.parametrize("n", [1, 31, 255, 256, 257, 5000])
@pytest.mark.parametrize("table", TABLES, ids=["default", "bytes", "wide"])
@pytest.mark.parametrize("copies", [False, True])
def test_queries_equal_the_oracle(forms, n, table, copies, monkeypatch):
    import torch

    if copies:  # host arrays uploaded, not read in place
        monkeypatch.setenv("ECHO_TEST_COPY_INPUTS", "1")

    q = _queries(np.random.default_rng(n), n, FORMS[forms])
    want = _want(q, table)
    fields = [(q.cc_type, np.uint8), (q.cc_algo, np.uint8), (q.nbytes, np.int64), (q.n_ranks, np.int32), (q.n_nodes, np.int32)]
    fields += [(x, np.float64) for x in (q.alpha_ns, q.bw_intra, q.lat_intra, q.bw_inter, q.lat_inter, q.delta)]
    host = [np.ascontiguousarray(x, dt) for x, dt in fields]
    tab = [np.array(x, np.int64) for x in table] if table else None
    last = (len(tab[0]), tab[0].ctypes.data, tab[1].ctypes.data) if tab else (0, None, None)
    out = np.full(n, np.nan)
    with E.Echo(0) as e:
        d = E.CCQueryDesc(n, *[h.ctypes.data for h in host], *last)
        assert e.lib.echo_cc_query(e.h, C.byref(d), C.c_void_p(out.ctypes.data)) == 0
    assert np.array_equal(out, want)
    dev = [torch.from_numpy(h).cuda() for h in host]
    d = E.CCQueryDesc(n, *[t.data_ptr() for t in dev], *last)
    into = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
    lib = E.load_library()
    for t in (into, dev[5]):  # (dev[5]: the start-up costs, overwritten by the results)
        assert lib.echo_cc_query_noalloc(C.byref(d), C.c_void_p(t.data_ptr()),
                                         C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
        assert np.array_equal(t.cpu().numpy(), want)


def test_a_chunk_times_the_ranks_beyond_64_bits():
    # 12 ranks with chunks of 2^60 bytes: every message is one round, also where the 64-bit product is negative
    size, N = (1 << 62) + (1 << 61), 12
    prm = [7.0, 3.0, 11.0, 5.0, 13.0, 0.25]
    host = [np.array([1], np.uint8), np.array([0], np.uint8), np.array([size]), np.array([N], np.int32), np.array([1], np.int32)]
    host += [np.array([x]) for x in prm]
    most, chunk = np.array([(1 << 63) - 1]), np.array([1 << 60])
    out = np.zeros(1)
    with E.Echo(0) as e:
        d = E.CCQueryDesc(1, *[h.ctypes.data for h in host], 1, most.ctypes.data, chunk.ctypes.data)
        assert e.lib.echo_cc_query(e.h, C.byref(d), C.c_void_p(out.ctypes.data)) == 0
    assert out[0] == 7.0 + (N - 1) * (11.0 + float(size) / N / 3.0)


def test_parameters_uploaded_or_read_in_place(monkeypatch):
    c = W.GPTConfig(**{**W.config("tiny").__dict__, "fixed_scenario": False})
    g = W.build_gpt_graph(c)
    for S in (1, 7, 300):
        sc = W.make_scenarios(g, c, n_scen=S)
        want = oracle.compose(g, sc)
        for copies in (False, True):
            if copies:
                monkeypatch.setenv("ECHO_TEST_COPY_INPUTS", "1")
            else:
                monkeypatch.delenv("ECHO_TEST_COPY_INPUTS", raising=False)
            with E.Echo(0) as e:
                e.load_graph(g)
                e.load_scenarios(sc)
                e.estimate_collectives()
                e.compose()
                assert np.array_equal(e.read_makespan(), want.makespan)
                assert np.array_equal(e.read_times()[1], want.finish)
