"""Graphs whose distance rows do not fit the shared memory of the static search: one source
at a time, its row there with a mask bit per vertex, or in D.  Sampled rows (d and sigma bit
for bit, delta within |err| <= 1e-9 * max(1, |x|)) of the static state and after updates."""
import numpy as np
import pytest

from paper_1311_2147_gb300 import binding, synth
from tests.parity_util import compare_rows

pytestmark = pytest.mark.gpu

WIDE = 1 << 31   # n of these do not fit 31 bits: the search runs in 64

CASES = [
    # (n, distances, directed, largest weight)
    (20000, "i64", True, WIDE),      # one source, row in shared memory
    (28001, "i64", False, WIDE),     # row in D
    (29100, "i32", True, 50),        # one source, 32-bit row
    (32768, "i64", True, 50),        # 64-bit distances searched in 32
    (32768, "i32", False, 50),
    (32768, "i64", True, WIDE),
]


@pytest.mark.parametrize("n,dist,directed,whi", CASES)
def test_large(n, dist, directed, whi):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = synth.erdos_renyi(n, (4 if directed else 2) * n, 1, whi, n, directed=directed)
    h = binding.BCGraph(g, dist=dist)
    rng = np.random.default_rng(n)
    rows = [0, n - 1] + rng.integers(0, n, 6).tolist()
    compare_rows(h, g, rows, bc_too=False, label=f"n={n} {dist} static")
    ups = synth.update_stream(g, 1, 1, 1, n + 1, 1, whi, kmin=2, kmax=4)
    rc, done = h.bc_apply_updates(ups)
    assert rc == binding.BC_OK and done == len(ups), h.last_error()
    compare_rows(h, synth.apply_updates(g, ups), rows, bc_too=False, label=f"n={n} {dist} updated")
    h.close()
