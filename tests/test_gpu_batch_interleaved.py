"""Two live batches of different graph sizes called in turn: what one batch's launch shape
sets on a kernel must not reach the other's launches.  The larger batch is captured again
(another number of rounds) after the smaller one was configured, with every thread count of
an accumulation CTA; each graph bit for bit as alone."""
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


def _graphs(ns, seed):
    out = []
    for i, n in enumerate(ns):
        make = synth.barabasi_albert if i % 2 else synth.erdos_renyi_degree
        g = make(n, 4, 1, 50, seed + i)
        out.append((g, synth.update_stream(g, 3, 4, 0, seed + 100 + i, 1, 50)))
    return out


@pytest.mark.parametrize("threads", [128, 256, 512])
@pytest.mark.parametrize("dist", ["i32", "i64"])
def test_two_batches_in_turn(dist, threads):
    fams = {"large": _graphs([2048, 1500], 11), "small": _graphs([64, 200], 21)}
    hs = {k: [binding.BCGraph(g, dist=dist) for g, _ in fam] for k, fam in fams.items()}
    bs = {k: binding.BCBatch(v) for k, v in hs.items()}
    for b in bs.values():
        b.bc_batch_set_tiles([4, 8, 8, 0, 4, 0, threads])
    at = {"large": 0, "small": 0}
    for k, rounds in [("large", 2), ("small", 2), ("large", 3), ("small", 1), ("large", 1), ("small", 3)]:
        part = [ups[at[k]:at[k] + rounds] for _, ups in fams[k]]
        rc, done = bs[k].bc_batch_apply(part)
        assert rc == binding.BC_OK, bs[k].last_error()
        assert done.tolist() == [rounds] * len(part)
        at[k] += rounds
    for k, fam in fams.items():
        for (g, ups), m in zip(fam, hs[k]):
            a = binding.BCGraph(g, dist=dist)
            rc, done = a.bc_apply_updates(ups[:at[k]])
            assert rc == binding.BC_OK and done == at[k]
            for x, y in zip(a.bc_get_rows(), m.bc_get_rows()):
                assert np.array_equal(x, y), f"{k} n={g.n}"
            assert np.array_equal(a.bc_get_scores(), m.bc_get_scores()), f"{k} n={g.n}"
            a.close()
    for b in bs.values():
        b.close()
