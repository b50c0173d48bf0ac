"""The batch autotuner times no value of a place in the launch shape that no kernel launch
reads (a timed value consumes updates of the caller's stream)."""
import glob
import re

from paper_1311_2147_gb300 import autotune, build


def test_no_candidates_for_an_unused_place():
    text = open(build.CSRC + "/bc_api.cu").read()
    body = text[text.index("int bc_batch_set_tiles("):text.index("int bc_batch_apply(")]
    kept = re.findall(r"b->L\.(\w+) = tiles\[(\d)\]", body)
    kernels = "".join(open(f).read() for f in glob.glob(build.CSRC + "/k_*.cu"))
    read = {int(i) for name, i in kept if re.search(r"\bL\." + name + r"\b", kernels)}
    assert read
    for i, values in enumerate(autotune.CANDIDATES):
        assert len(values) == 1 or i in read, i
