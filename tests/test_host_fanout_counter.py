"""The fan-out's control kernels add to the count of finished objectives, so none of their
blocks may decide by it: another block of the same launch may have changed it."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2307_03466_gb300", "csrc",
                   "fanout.cu")


def kernels(text):
    """name -> body of every __global__ function."""
    out = {}
    for m in re.finditer(r"__global__ void[^{;]*?(k_\w+)\([^{;]*\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        out[m.group(1)] = text[m.end():i]
    return out


def test_kernels_that_count_finished_objectives_do_not_read_the_count():
    with open(SRC) as f:
        bodies = kernels(f.read())
    writers = [k for k, b in bodies.items() if re.search(r"atomicAdd\(F\.n_done", b)]
    assert sorted(writers) == ["k_fcheck_control", "k_fstep_control"]
    for k in writers:
        assert not re.search(r"\*F\.n_done\b|fan_over\(", bodies[k]), k
