"""Static searches: dense graphs, whose searches are restricted to arcs no longer than the
paths over each vertex's lightest arcs (equal weights, few lightest arcs, wide weights,
unreachable pairs among the light arcs), and vertex counts around the search's groups of
sources, against the oracle (d and sigma bit for bit, delta and BC within
|err| <= 1e-9 * max(1, |x|))."""
import numpy as np
import pytest

from paper_1311_2147_gb300 import binding, synth
from tests.parity_util import compare_full

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    binding.load()


def _two_cliques(n):
    """Two complete halves joined by heavy arcs only, so that light paths miss the other half."""
    g = synth.complete_directed(n, 1, 9, 6)
    far = (g.src < n // 2) != (g.dst < n // 2)
    return synth.Graph(n, True, g.src, g.dst, np.where(far, 1000 + g.w, g.w))


DENSE = {
    "random": (lambda: synth.complete_directed(130, 1, 130 * 130, 5), "i64"),
    "equal": (lambda: synth.complete_graph(90, True, 4), "i32"),
    "two-values": (lambda: synth.complete_directed(97, 1, 2, 7), "i32"),
    "undirected": (lambda: synth.erdos_renyi(100, 3000, 1, 40, 8, directed=False), "i32"),
    "wide": (lambda: synth.complete_directed(70, 1 << 40, (1 << 40) + 5000, 9), "i64"),
    "halves": (lambda: _two_cliques(80), "i64"),
}


@pytest.mark.parametrize("name", sorted(DENSE))
def test_dense(name):
    make, dist = DENSE[name]
    g = make()
    h = binding.BCGraph(g, dist=dist)
    compare_full(h, g, label=name)
    h.close()


@pytest.mark.parametrize("dist", ["i32", "i64"])
@pytest.mark.parametrize("n", [2, 151, 153, 305, 620])
def test_groups_of_sources(n, dist):
    g = synth.erdos_renyi(n, min(3 * n, n * (n - 1)), 1, 1 << 27 if dist == "i64" else 30, 50 + n, directed=True)
    h = binding.BCGraph(g, dist=dist)
    compare_full(h, g, label=f"n={n} {dist}")
    h.close()
