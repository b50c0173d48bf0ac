"""The walked pair corrections of a batch: each graph must get, bit for bit, what the same
updates give it alone with the same options -- graphs that walk beside graphs corrected by
the column test, directed ones, one whose rows all take the dense tables, and an update of
more than 32 edges, which is corrected by the column test in a graph that walks."""
import numpy as np
import pytest

from paper_1311_2147_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    binding.load()


def _member(i):
    """(graph, updates, options) of the i-th graph."""
    opts = []
    if i == 0:      # long paths: rows with up to 128 targets, tables outgrown
        g = synth.path_graph(300, False, 1)
        return g, [("edge", 0, 299, 1), ("edge", 100, 200, 3), ("edge", 50, 250, 1)], opts
    if i == 1:      # two vertices
        return synth.path_graph(2, False, 9), [("edge", 0, 1, 4), ("edge", 0, 1, 2)], [("walk_cap", 0)]
    if i == 6:
        g = synth.erdos_renyi(60, 400, 1, 20, 506, directed=True)
        return g, synth.update_stream(g, 2, 2, 2, 606, 1, 20, kmin=1, kmax=4), opts
    g = (synth.barabasi_albert(90 + 61 * i, 4, 1, 6, 500 + i) if i % 2
         else synth.erdos_renyi(77 + 40 * i, 400 + 100 * i, 1, 9, 500 + i, directed=False))
    ups = synth.update_stream(g, 2, 2, 2, 600 + i, 1, 6, kmin=1, kmax=5)
    if i == 2:
        em = synth.EdgeMap.of(synth.apply_updates(g, ups))
        far = [x for x in range(g.n - 1, 0, -1) if x != 5 and em.get(x, 5) is None][:40]
        ups.append(("vertex", 5, [(x, 2, 0) for x in far]))
        ups += synth.update_stream(synth.apply_updates(g, ups), 1, 1, 1, 700, 1, 6, kmin=1, kmax=5)
    if i == 3:
        opts.append(("pair_walk", 0))
    if i == 4:
        opts.append(("walk_cap", 0))
    return g, ups, opts


@pytest.mark.parametrize("dist", ["i32", "i64"])
def test_batch_equals_alone(dist):
    members = [_member(i) for i in range(8)]
    hs = []
    for _ in range(2):
        hs.append([])
        for g, _, opts in members:
            h = binding.BCGraph(g, dist=dist)
            for name, value in opts:
                h.bc_set_option(name, value)
            hs[-1].append(h)
    alone, together = hs
    b = binding.BCBatch(together)
    for part in (slice(0, 2), slice(2, None)):   # two calls of different rounds
        rc, done = b.bc_batch_apply([ups[part] for _, ups, _ in members])
        assert rc == 0
        for h, (_, ups, _) in zip(alone, members):
            rc, _ = h.bc_apply_updates(ups[part])
            assert rc == 0
        for i, (x, y) in enumerate(zip(alone, together)):
            for p, q in zip(x.bc_get_rows() + (x.bc_get_scores(),), y.bc_get_rows() + (y.bc_get_scores(),)):
                assert np.array_equal(p, q), f"graph {i}"
    for i, (x, y) in enumerate(zip(alone, together)):
        ix, iy = x.bc_get_info(), y.bc_get_info()
        for k in ("pair_rows", "pair_targets", "walk_pairs", "walk_vertices", "walk_arcs", "rows_full"):
            assert ix[k] == iy[k], f"graph {i}: {k}"
    assert together[0].bc_get_info()["walk_pairs"] > 0 and together[3].bc_get_info()["walk_pairs"] == 0
    b.close()
