"""The forms of the dependency accumulation (dev_accum_source), each where it can go wrong,
statically and after updates that re-accumulate every changed row, against the oracle (d
and sigma bit for bit, delta and BC within |err| <= 1e-9 * max(1, |x|)):

* more DAG arcs than the pool holds (complete bipartite, unit weights);
* more levels than fit beside the other arrays (a path of 700 vertices);
* vertices with 30, 31, 32 and several hundred DAG out-arcs (stars);
* int64 distances past 31 bits (read from memory) next to ones that fit;
* the superset's slot mask, and the per-vertex cells, in the work space.
"""
import numpy as np
import pytest

from paper_1311_2147_gb300 import binding, synth
from tests.parity_util import compare_full, compare_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    binding.load()


def _of(n, directed, edges):
    e = np.array(edges, dtype=np.int64)
    return synth.Graph(n, directed, e[:, 0].astype(np.int32), e[:, 1].astype(np.int32), e[:, 2])


def _bipartite(k, w):
    return _of(2 * k, False, [(a, k + b, w) for a in range(k) for b in range(k)])


def _stars(sizes, w):
    """Stars of the given leaf counts, their centres in a chain."""
    edges, at, centres = [], 0, []
    for size in sizes:
        centres.append(at)
        edges += [(at, at + 1 + i, w) for i in range(size)]
        at += 1 + size
    edges += [(a, b, w) for a, b in zip(centres, centres[1:])]
    return _of(at, False, edges)


def _scaled(g, f):
    return synth.Graph(g.n, g.directed, g.src, g.dst, g.w * f)


CASES = {
    "ties": (lambda: _bipartite(90, 2), "i32", [("edge", 0, 1, 3), ("edge", 0, 95, 1)]),
    "ties-i64": (lambda: _bipartite(40, 2), "i64", [("edge", 3, 1, 2), ("edge", 5, 60, 1)]),
    "levels": (lambda: synth.path_graph(700, False, 2), "i32", [("edge", 100, 101, 1), ("edge", 10, 650, 1270)]),
    "big": (lambda: _stars([30, 31, 32, 300], 3), "i32", [("edge", 1, 40, 1), ("edge", 0, 31, 1)]),
    "wide": (lambda: _scaled(synth.erdos_renyi(90, 300, 1, 50, 5, directed=True), 1 << 33), "i64",
             [("edge", 1, 2, 7), ("vertex", 5, [(6, 1 << 33, 0), (7, 9, 1)])]),
    "wide-edge": (lambda: _of(5, True, [(0, 1, (1 << 31) - 2), (1, 2, 1), (2, 3, 1), (3, 4, 5), (0, 4, 1 << 40)]), "i64",
                  [("edge", 0, 2, (1 << 31) - 1)]),
    "one": (lambda: synth.Graph(1, True, np.zeros(0, np.int32), np.zeros(0, np.int32), np.zeros(0, np.int64)), "i32", []),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_small_forms(name):
    make, dist, ups = CASES[name]
    g = make()
    h = binding.BCGraph(g, dist=dist)
    if not g.directed:
        h.bc_set_option("pair_updates", 0)
    compare_full(h, g, label=f"{name} static")
    for i, up in enumerate(ups):
        rc, done = h.bc_apply_updates([up])
        assert rc == binding.BC_OK and done == 1, (name, up, h.last_error())
        compare_full(h, synth.apply_updates(g, ups[: i + 1]), label=f"{name} after {i + 1}")
    h.close()


@pytest.mark.parametrize("name", ["mask", "cells"])
def test_arrays_in_the_work_space(name):
    if name == "mask":
        n = 1100   # a complete graph of equal weights keeps all its arcs in the superset
        a, b = np.nonzero(~np.eye(n, dtype=bool))
        g = synth.Graph(n, True, a.astype(np.int32), b.astype(np.int32), np.full(a.shape[0], 2, np.int64))
        ups = [("edge", 3, 9, 1)]
    else:
        g = synth.erdos_renyi(6001, 13000, 1, 9, 17, directed=True)
        ups = synth.update_stream(g, 1, 1, 1, 18, 1, 9, kmin=2, kmax=3)
    h = binding.BCGraph(g)
    rc, done = h.bc_apply_updates(ups)
    assert rc == binding.BC_OK and done == len(ups), h.last_error()
    compare_rows(h, synth.apply_updates(g, ups), [0, 3, g.n // 2, g.n - 1], label=name)
    h.close()
