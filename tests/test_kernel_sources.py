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


def test_only_the_copy_of_the_inputs_is_chained_to_the_work_ahead_of_a_call():
    """The launches of a forward call request weights ahead of their own waits, so the first of them starts when all that the
    caller enqueued before has finished.  The copy may start early: it waits before its first access."""
    runtime = _code("runtime.cu")
    uses = re.findall(r"[^;{}]*\bmay_open\(st\)[^;{}]*;", runtime)
    assert len(uses) == 1 and "return launch_copy2(" in uses[0], uses
    run_ops = runtime[runtime.index("static int run_ops("):]
    run_ops = run_ops[:run_ops.index("\n}")]
    assert "bool chained = false;\n  for (" in run_ops
    assert re.findall(r"\bissue\((.*)\)", run_ops) == ["pl, pl->ops[i], st, chained"]
    copy = _code("elementwise.cu")
    copy = copy[copy.index("copy2_kernel(uint8_t* dst0"):]
    assert copy[copy.index("{") + 1:].split(";")[0].strip() == "grid_dep_wait()"
