"""Dependencies far below one: where pairs have 3^k shortest paths, a vertex on one of them
has a dependency of about 3^-k.  Updates bring such a vertex onto the shortest paths; the
corrected and the re-accumulated rows, and BC, keep its relative accuracy.

Tolerance: a result goes through at most a few hundred float-float operations, each with a
relative error of a few units of 2^-46 (ff.cuh), all on terms of one sign for the vertices
compared (new on the paths, so nothing cancels): 512 * 4 * 2^-46 = 2.9e-11.  BC's change keeps
each of these to 2^-112, far below that of the entries here."""
import numpy as np
import pytest

from oracle import oracle
from paper_1311_2147_gb300 import binding, synth

pytestmark = pytest.mark.gpu

RTOL = 512 * 4 * 2.0 ** -46


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    binding.load()


def chain(k, tail, directed):
    """a_0 .. a_k, each joined to the next over three vertices (3^k shortest paths of length
    2k), a path of `tail` vertices before a_0 and after a_k, and a vertex x whose arcs to a_0
    and a_k are too long to matter.  Returns (graph, x, a_0, a_k)."""
    e = []
    for i in range(k):
        for b in range(4 * i + 1, 4 * i + 4):
            e += [(4 * i, b, 1), (b, 4 * i + 4, 1)]
    end, at = 4 * k, 4 * k + 1
    for i in range(tail):
        e += [(end if i == 0 else at + i - 1, at + i, 1)]
    at += tail
    for i in range(tail):
        e += [(at + i, 0 if i == 0 else at + i - 1, 1)]
    x = at + tail
    e += [(0, x, 5 * k), (x, end, 5 * k)]
    src, dst, w = (np.array(c, np.int64) for c in zip(*e))
    return synth.Graph(x + 1, directed, src.astype(np.int32), dst.astype(np.int32), w), x, 0, end


def check(h, g, x, a0, label):
    st = oracle.brandes(g)
    d, s, dl = h.bc_get_rows()
    assert np.array_equal(d, st.D) and np.array_equal(s, st.SIG), label
    got, exp = dl[:, x], st.DEL[:, x]
    assert exp[a0] > 0
    assert bool(np.all(np.abs(got - exp) <= RTOL * exp)), f"{label}: dependency {got[a0]} expected {exp[a0]}"
    bc = h.bc_get_scores()[x]
    assert abs(bc - st.BC[x]) <= RTOL * st.BC[x], f"{label}: BC {bc} expected {st.BC[x]}"


@pytest.mark.parametrize("dist", ["i32", "i64"])
@pytest.mark.parametrize("form", ["walk", "dense", "column-test", "full", "batch"])
@pytest.mark.parametrize("k", [8, 16, 25])
def test_undirected(k, form, dist):
    g, x, a0, ak = chain(k, 5, False)
    h = binding.BCGraph(g, dist=dist)
    if form == "dense":
        h.bc_set_option("walk_cap", 0)
    elif form == "column-test":
        h.bc_set_option("pair_walk", 0)
    elif form == "full":
        h.bc_set_option("pair_updates", 0)
    ups = [("edge", a0, x, k), ("edge", x, ak, k)]
    if form == "batch":
        batch = binding.BCBatch([h])
        rc, _ = batch.bc_batch_apply([ups])
    else:
        rc, _ = h.bc_apply_updates(ups)
    assert rc == binding.BC_OK
    check(h, synth.apply_updates(g, ups), x, a0, f"k={k} {form} {dist}")
    h.close()


@pytest.mark.parametrize("k", [8, 16, 25])
def test_directed(k):
    g, x, a0, ak = chain(k, 5, True)
    h = binding.BCGraph(g, dist="i32")
    ups = [("edge", a0, x, k), ("edge", x, ak, k)]
    rc, _ = h.bc_apply_updates(ups)
    assert rc == binding.BC_OK
    check(h, synth.apply_updates(g, ups), x, a0, f"k={k}")
    h.close()
