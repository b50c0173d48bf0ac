"""Rows of the state are padded to a multiple of eight entries: vertex counts on both
sides of the padding, of a 32-bit change-map word and of a rank-1 column chunk, against
the oracle after a stream of edge and vertex updates (d and sigma bit for bit, delta and
BC within |err| <= 1e-9 * max(1, |x|))."""
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


@pytest.mark.parametrize("directed", [True, False], ids=["directed", "undirected"])
@pytest.mark.parametrize("dist", ["i32", "i64"])
@pytest.mark.parametrize("n", [7, 8, 9, 31, 33, 255, 1025])
def test_padded_rows(n, dist, directed):
    g = synth.erdos_renyi(n, 2 * n, 1, 9, 40 + n, directed=directed)
    ups = synth.update_stream(g, 3, 3, 3, 41 + n, 1, 9, kmin=1, kmax=3)
    h = binding.BCGraph(g, dist=dist)
    rc, done = h.bc_apply_updates(ups)
    assert rc == binding.BC_OK and done == len(ups), h.last_error()
    compare_full(h, synth.apply_updates(g, ups), label=f"n={n} {dist}")
    h.close()
