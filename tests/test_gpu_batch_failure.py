"""A batch call that fails after its updates entered the host weights: the graphs that had
updates are poisoned, so that their weights and their state on the device cannot differ
unnoticed.  The failure is made on the host: the batch's stream is being captured already,
so the batch cannot capture its rounds."""
import pytest

from paper_1311_2147_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def test_failed_capture_poisons_the_graphs_with_updates():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = synth.erdos_renyi_degree(100, 4, 10, 50, 3)
    ups = synth.update_stream(g, 2, 2, 0, 4, 2, 50)
    torch.zeros(1, device="cuda")
    with_ups, without = binding.BCGraph(g), binding.BCGraph(g)
    st = torch.cuda.Stream()
    batch = binding.BCBatch([with_ups, without], stream=st.cuda_stream)
    rc, _ = batch.bc_batch_apply([ups[:1], []])
    assert rc == binding.BC_OK, batch.last_error()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        graph.capture_begin(capture_error_mode="relaxed")
        rc, _ = batch.bc_batch_apply([ups[1:3], []])   # another number of rounds: a capture of its own
        try:
            graph.capture_end()
        except RuntimeError:
            pass
    assert rc == binding.BC_ERR_CUDA
    assert with_ups.lib.bc_get_scores(with_ups.h, None) == binding.BC_ERR_POISONED
    u, v, w = ups[1][1:]
    assert with_ups.bc_apply_edge_update(u, v, w - 1) == binding.BC_ERR_POISONED
    rc, done = without.bc_apply_updates(ups)   # no update of its own in the failed call
    assert rc == binding.BC_OK and done == len(ups), without.last_error()
