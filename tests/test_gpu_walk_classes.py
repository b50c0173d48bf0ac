"""The classes of the walked pair corrections: a row's result must not depend on the table
that it ran in.

The option "walk_cap" bounds the entries of the shared-memory tables: 0 sends every row to
the dense arrays in device memory, 40 all but the smallest to a CTA or to those, the default
leaves each row where it belongs.  Sums are integers, so the three must agree bit for bit
after every update; against the column test, dependencies within 1e-9 * max(1, |x|).
An update of more than 32 edges in between is corrected by the column test.
"""
import numpy as np
import pytest

from paper_1311_2147_gb300 import binding, synth
from tests.parity_util import close, compare_full

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    binding.load()


def _cases():
    p = synth.path_graph(300, False, 1)      # up to 128 targets a row, on paths of hundreds of vertices
    yield "path", p, [("edge", 0, 299, 1), ("edge", 100, 200, 3), ("vertex", 50, [(250, 1, 0), (120, 2, 0)])]
    e = synth.erdos_renyi(129, 900, 1, 2, 77, directed=False)    # small weights: many parents a vertex
    yield "ties", e, synth.update_stream(e, 6, 4, 4, 78, 1, 2, kmin=2, kmax=5)
    b = synth.barabasi_albert(700, 6, 1, 4, 79)                  # hubs, ties
    ups = synth.update_stream(b, 5, 5, 4, 80, 1, 4, kmin=2, kmax=6)
    em = synth.EdgeMap.of(synth.apply_updates(b, ups))
    far = [x for x in range(b.n - 1, 0, -1) if x != 300 and em.get(x, 300) is None][:40]
    ups += [("vertex", 300, [(x, 2, 0) for x in far])]
    ups += synth.update_stream(synth.apply_updates(b, ups), 2, 2, 2, 81, 1, 4, kmin=2, kmax=6)
    yield "hubs", b, ups


@pytest.mark.parametrize("dist", ["i32", "i64"])
@pytest.mark.parametrize("which", [0, 1, 2])
def test_classes_agree(which, dist):
    label, g, ups = list(_cases())[which]
    hs = []
    for cap in (0, 40, None):
        h = binding.BCGraph(g, dist=dist)
        h.bc_set_option("pair_walk", 1)
        if cap is not None:
            h.bc_set_option("walk_cap", cap)
        hs.append(h)
    col = binding.BCGraph(g, dist=dist)
    col.bc_set_option("pair_walk", 0)
    for i, up in enumerate(ups):
        for h in hs + [col]:
            rc, done = h.bc_apply_updates([up])
            assert rc == 0 and done == 1, (label, up, h.last_error())
        want = hs[-1].bc_get_rows() + (hs[-1].bc_get_scores(),)
        for h in hs[:-1]:
            got = h.bc_get_rows() + (h.bc_get_scores(),)
            for x, y in zip(got, want):
                assert np.array_equal(x, y), f"{label}: update {i}"
        d, s, dl = col.bc_get_rows()
        assert np.array_equal(d, want[0]) and np.array_equal(s, want[1]), f"{label}: update {i}"
        ok, worst = close(dl, want[2])
        assert ok, f"{label}: dependencies, update {i} ({worst:.3g} x tol)"
    assert hs[-1].bc_get_info()["walk_pairs"] > 0
    compare_full(hs[-1], synth.apply_updates(g, ups), label=label)
