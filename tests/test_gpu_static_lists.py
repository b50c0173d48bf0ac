"""Static searches whose rounds change few vertices (these go over lists of them) and pass
between such rounds and rounds over all arcs: paths, cycles, grids, hubs along a path whose
leaves do not fit a list.  Against the oracle (d and sigma bit for bit, delta and BC within
|err| <= 1e-9 * max(1, |x|)), through bc_init_static and, where it fits, the entry point
that allocates nothing."""
import numpy as np
import pytest

from paper_1311_2147_gb300 import binding, synth
from tests.parity_util import close, compare_full, compare_rows
from tests.test_zz_no_alloc import _call

pytestmark = pytest.mark.gpu


def _grid(rows, cols, directed, whi):
    at = np.arange(rows * cols).reshape(rows, cols)
    src = np.concatenate([at[:, :-1].ravel(), at[:-1].ravel()])
    dst = np.concatenate([at[:, 1:].ravel(), at[1:].ravel()])
    w = synth.Rng(rows).uniform_int(1, whi, src.size)
    return synth.Graph(rows * cols, directed, src.astype(np.int32), dst.astype(np.int32), np.asarray(w, np.int64))


def _hubs(n, leaves):
    """A path with two hubs of `leaves` leaves each at a third and two thirds of it."""
    e = [(i, i + 1) for i in range(n - 1)]
    for h, hub in enumerate((n // 3, 2 * n // 3)):
        e += [(hub, n + h * leaves + i) for i in range(leaves)]
    src, dst = (np.array(c, np.int32) for c in zip(*e))
    return synth.Graph(n + 2 * leaves, False, src, dst, np.full(len(e), 3, np.int64))


GRAPHS = {
    "path": (lambda w: synth.path_graph(700, w=w)),
    "grid-large": (lambda w: _grid(40, 60, False, min(w, 1 << 31))),
    "cycle": (lambda w: synth.cycle_graph(401, True, w=w)),
    "grid": (lambda w: _grid(9, 50, False, 10)),
    "grid-directed": (lambda w: _grid(30, 30, True, 1 << 20)),
    "hubs": (lambda w: _hubs(300, 600)),
}


@pytest.mark.parametrize("dist,w", [("i32", 2), ("i64", 2), ("i64", 1 << 40)])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_lists(name, dist, w):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = GRAPHS[name](w)
    h = binding.BCGraph(g, dist=dist)
    st = compare_full(h, g, label=f"{name} {dist}")
    h.close()
    if g.n <= 512:
        flags = (binding.BC_DIRECTED if g.directed else binding.BC_UNDIRECTED) | (
            binding.BC_DIST_I32 if dist == "i32" else binding.BC_DIST_I64)
        rc, got = _call(binding.load(), torch, g, flags)
        assert rc == binding.BC_OK
        ok, worst = close(got, st.BC)
        assert ok, f"{name} {dist}: worst error {worst:.3g} x tolerance"


def test_dense_and_large():
    """One source per CTA over arcs in no order (a dense graph's light and filtered ones)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = synth.erdos_renyi(20000, 50 * 20000, 1, 1 << 31, 9, directed=True)
    h = binding.BCGraph(g, dist="i64")
    compare_rows(h, g, [0, 7777, 19999], bc_too=False, label="dense n=20000")
    h.close()
