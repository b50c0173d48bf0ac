"""Accumulations of DAGs with more arcs than the pool holds, whose heads are read off the
masks and the superset, and of vertices with many DAG out-arcs, placed by a warp: stars, hubs
of a few thousand arcs, equal weights.  Against the oracle (d and sigma bit for bit, delta and
BC within |err| <= 1e-9 * max(1, |x|)); and a graph whose pool overflows alone but not beside
a larger one in a batch, bit for bit."""
import numpy as np
import pytest

from paper_1311_2147_gb300 import binding, synth
from tests.parity_util import compare_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    binding.load()


def _hub(n, k, directed, w):
    """A path with a hub of k leaves in the middle; the leaves' own arcs lead on to a ring."""
    leaves = list(range(n - k, n))
    mid = (n - k) // 2
    e = [(i, i + 1, 2) for i in range(n - k - 1)] + [(mid, x, w + i % 3) for i, x in enumerate(leaves)]
    e += [(leaves[i], leaves[i + 1], 1) for i in range(0, k - 1, 2)]
    src, dst, ww = (np.array(c, np.int64) for c in zip(*e))
    return synth.Graph(n, directed, src.astype(np.int32), dst.astype(np.int32), ww)


GRAPHS = {
    "star": lambda: synth.star_graph(2500, 3),
    "hub-2000": lambda: _hub(3000, 2000, False, 5),
    "hub-directed": lambda: _hub(2200, 1500, True, 1 << 35),
    "hub-255": lambda: _hub(900, 255, False, 4),
    "hub-256": lambda: _hub(900, 256, False, 4),
    "hub-700": lambda: _hub(2600, 700, False, 5),
    "equal-ba": lambda: synth.barabasi_albert(1500, 8, 4, 4, 3),
    "equal-er": lambda: synth.erdos_renyi(1100, 12000, 2, 2, 4, directed=True),
    "two-values": lambda: synth.complete_directed(150, 1, 2, 7),
}


@pytest.mark.parametrize("dist", ["i32", "i64"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_against_oracle(name, dist):
    g = GRAPHS[name]()
    if dist == "i32" and int(g.w.max()) >= 1 << 31:
        pytest.skip("weights need 64-bit distances")
    h = binding.BCGraph(g, dist=dist)
    rng = np.random.default_rng(1)
    rows = [0, g.n // 2, g.n - 1] + rng.integers(0, g.n, 5).tolist()
    compare_rows(h, g, rows, label=f"{name} {dist}")
    ups = [("edge", int(g.src[i]), int(g.dst[i]), int(g.w[i]) // 2) for i in (g.m - 1, g.m // 2, g.m // 5) if g.w[i] > 1]
    rc, done = h.bc_apply_updates(ups)
    assert rc == binding.BC_OK and done == len(ups), h.last_error()
    compare_rows(h, synth.apply_updates(g, ups), rows, label=f"{name} {dist} updated")
    h.close()


@pytest.mark.parametrize("pairs", [1, 0])
def test_pool_and_masks_bit_for_bit(pairs):
    small = synth.barabasi_albert(700, 8, 6, 6, 5)      # more DAG arcs than its own pool holds
    large = synth.barabasi_albert(2600, 2, 1, 1000, 6)  # whose layout the batch takes
    ups = [("edge", int(a), int(b), 5) for a, b in zip(small.src[::900], small.dst[::900])]
    alone = binding.BCGraph(small, dist="i32")
    hs = [binding.BCGraph(small, dist="i32"), binding.BCGraph(large, dist="i32")]
    for h in [alone] + hs[:1]:
        h.bc_set_option("pair_updates", pairs)
    assert alone.bc_apply_updates(ups) == (binding.BC_OK, len(ups))
    batch = binding.BCBatch(hs)
    rc, _ = batch.bc_batch_apply([ups, []])
    assert rc == binding.BC_OK, batch.last_error()
    for x, y in zip(alone.bc_get_rows(), hs[0].bc_get_rows()):
        assert np.array_equal(x, y)
    assert np.array_equal(alone.bc_get_scores(), hs[0].bc_get_scores())
    compare_rows(alone, synth.apply_updates(small, ups), [0, 350, 699])
