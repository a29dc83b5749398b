"""Host arrays at any byte address: kernels read a caller's arrays in place only where every element is aligned
(``csrc/echo_align.h``, compiled here with g++), and calls with arrays that are not give the same results as with
aligned ones, as their copies do."""
import ctypes as C
import dataclasses
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_2412_12487_gb300 import build as B
from paper_2412_12487_gb300 import echo as E
from paper_2412_12487_gb300 import workloads as W

MAIN = r"""
#include "echo_align.h"
#include <stdio.h>
int main() {
  alignas(16) char b[64];
  using echo::elements_aligned;
  int bad = 0;
  for (size_t size : {1, 4, 8})
    for (int at = 0; at < 16; ++at) {
      bad += elements_aligned(size, {b + at}) != (at % size == 0);
      for (int k = 0; k < 3; ++k) {  // any one of several decides
        const char *p[3] = {b, b + 16, b + 32};
        p[k] += at;
        bad += elements_aligned(size, {p[0], p[1], p[2]}) != (at % size == 0);
      }
    }
  bad += !elements_aligned(8, {});
  return bad;
}
"""


def test_alignment_of_every_array_decides(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(B.ROOT, B.CSRC), str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def _at(x, offset):
    """The array x at an address that is `offset` bytes past a multiple of 16."""
    x = np.ascontiguousarray(x)
    raw = np.empty(x.nbytes + 32, np.uint8)
    first = (offset - raw.ctypes.data) % 16
    y = raw[first:first + x.nbytes].view(x.dtype).reshape(x.shape)
    y[...] = x
    assert y.ctypes.data % 16 == offset
    return y


@pytest.mark.gpu
@pytest.mark.parametrize("offset", [0, 1, 4, 8])
@pytest.mark.parametrize("which", ["alpha_ns", "bw_intra", "lat_intra", "bw_inter", "lat_inter", "delta", "slowdown", "dur"])
def test_scenarios_from_unaligned_arrays(which, offset):
    c = W.GPTConfig(**{**W.config("tiny").__dict__, "fixed_scenario": False})
    g = W.build_gpt_graph(c)
    sc = W.make_scenarios(g, c, n_scen=5)
    want = oracle.compose(g, sc)
    with E.Echo(0) as e:
        e.load_graph(g)
        e.load_scenarios(dataclasses.replace(sc, **{which: _at(getattr(sc, which), offset)}))
        e.estimate_collectives()
        e.compose()
        assert np.array_equal(e.read_times()[1], want.finish)


@pytest.mark.gpu
@pytest.mark.parametrize("offset", [0, 1, 2, 4, 8])
@pytest.mark.parametrize("which", ["nbytes", "n_ranks", "n_nodes", "alpha_ns", "bw_intra", "lat_intra", "bw_inter", "lat_inter", "delta"])
def test_queries_from_unaligned_arrays(which, offset):
    q = W.make_cc_queries(300, seed=5)
    with E.Echo(0) as e:
        want = e.cc_query(q)
        got = e.cc_query(dataclasses.replace(q, **{which: _at(getattr(q, which), offset)}))
        out = _at(np.zeros(q.n), offset)
        keep = [np.ascontiguousarray(getattr(q, f.name)) for f in dataclasses.fields(q)]
        d = E.CCQueryDesc(q.n, *[x.ctypes.data for x in keep], 0, None, None)
        assert e.lib.echo_cc_query(e.h, C.byref(d), C.c_void_p(out.ctypes.data)) == 0
    assert np.array_equal(got, want) and np.array_equal(out, want)
