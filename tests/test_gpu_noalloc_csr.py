"""bc_static_scores_noalloc refuses offsets that do not cover the arcs: slots outside them
would hold arcs of an earlier call, of a larger graph here."""
import pytest

from oracle import oracle
from paper_1311_2147_gb300 import binding, synth
from tests.parity_util import close
from tests.test_zz_no_alloc import _call, _device_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dist", [binding.BC_DIST_I32, binding.BC_DIST_I64])
@pytest.mark.parametrize("first,last", [(1, 0), (0, -1), (2, -3)])
def test_offsets_that_leave_slots_out(first, last, dist):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = binding.load()
    large = synth.erdos_renyi(500, 3000, 1, 20, 1, directed=True)
    small = synth.erdos_renyi(40, 300, 1, 20, 2, directed=True)
    flags = binding.BC_DIRECTED | dist
    assert _call(lib, torch, large, flags)[0] == binding.BC_OK
    inputs = _device_inputs(torch, small)
    inputs[0][0] += first
    inputs[0][-1] += last
    torch.cuda.synchronize()
    assert _call(lib, torch, small, flags, inputs)[0] == binding.BC_ERR_ARG
    rc, got = _call(lib, torch, small, flags)
    assert rc == binding.BC_OK
    ok, worst = close(got, oracle.brandes(small, want_rows=False).BC)
    assert ok, f"worst error {worst:.3g} x tolerance"
