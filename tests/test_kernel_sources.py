"""Rules of the chained launches that no result shows, checked on the kernels' sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_11136_b200", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_chained_kernels_wait_before_they_read_activations():
    """What an earlier launch wrote is visible to a chained kernel only behind griddepcontrol.wait: every
    call of grid_dep_wait() is a statement of its own, never one that a flag can skip, and in the GEMM's
    producer it stands before the first activation load."""
    calls = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        for m in re.finditer(r"([^;{}]*)\bgrid_dep_wait\(\)", _code(name)):
            before = m.group(1).strip()
            if before.startswith("using"):
                continue
            calls += 1
            assert before in ("", "__syncwarp()"), (name, before)
    assert calls >= 5
    gemm = _code("gemm.cu")
    producer = gemm[gemm.index("const int early = worker"):]
    assert producer.index("grid_dep_wait()") < producer.index("load_a(")
