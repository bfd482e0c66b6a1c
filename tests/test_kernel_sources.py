"""Rules of the chained launches that no result shows, checked on the kernels' sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_11136_b200", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _headers(code, at):
    """What opens the blocks around position `at`, innermost first."""
    out, depth = [], 0
    for i in range(at - 1, -1, -1):
        if code[i] == "}":
            depth += 1
        elif code[i] == "{" and depth:
            depth -= 1
        elif code[i] == "{":
            head = re.split(r"[{}]", code[:i])[-1]
            loop = head.rfind("for (")
            head = head[loop:] if loop >= 0 else head.split(";")[-1]
            out.append(" ".join(head.split()))
    return out


# What a wait for earlier launches stands under, with the reason why nothing of theirs is touched without it.
CONDITIONS = {
    "gemm.cu": {
        "if (early > 0)": 1,                              # the producer of a CTA without tiles loads nothing
        "if constexpr (!kRehearse<BN, PAIR>)": 1,         # epilogue, tiles that do not rehearse: before the first tile
        "if (dry)": 1,                                    # ... that do: at the end of the rehearsal, which is the first round
        "else": 1,                                        # the epilogue's role itself: a CTA without tiles waits behind the loop
    },
    "attention.cu": {
        "if (warp < 4)": 1,                               # producer and issuers
        "else": 1,                                        # softmax warps, instances that do not rehearse
        "if (REHEARSE && i == 0)": 1,                     # ... that do: before the first item
    },
}


def test_chained_kernels_wait_before_they_read_activations():
    """What an earlier launch wrote is visible to a chained kernel only behind griddepcontrol.wait: every call of
    grid_dep_wait() is a statement of its own, at the top of a kernel or under one of the conditions listed above,
    and in the GEMM's producer it stands before the first activation load."""
    free = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        code, under = _code(name), {}
        for m in re.finditer(r"([^;{}]*)\bgrid_dep_wait\(\)", code):
            before = m.group(1).strip()
            if before.startswith("using"):
                continue
            assert before in ("", "__syncwarp()"), (name, before)
            head = _headers(code, m.start(1))[0]
            if head == "else" or head.startswith(("if ", "for ", "while ")):
                under[head] = under.get(head, 0) + 1
            else:
                free += 1
        assert under == CONDITIONS.get(name, {}), name
    assert free >= 3
    gemm = _code("gemm.cu")
    producer = gemm[gemm.index("const int early = worker"):]
    assert producer.index("grid_dep_wait()") < producer.index("load_a(")


def test_rehearsals_touch_nothing_of_earlier_launches():
    """A rehearsal runs before the wait: of the statements of its round that reach outside the CTA or wait for something, each
    says that it is not for the rehearsal."""
    gemm = _code("gemm.cu")
    epilogue = gemm[gemm.index("const bool dry = ep.rehearsing();"):]
    epilogue = epilogue[:epilogue.index("if (dry) {")]
    epilogue = re.sub(r"for \([^{}\n]*\)", lambda m: m.group().replace(";", ","), epilogue)
    reaches = list(re.finditer(r"ep\.request\(|ep\.load_angles\(|__ldg\(|ld_f2\(|mbar_wait_warp\(|bulk_commit\(|tma_", epilogue))
    assert len(reaches) == 5
    for m in reaches:
        # the statement itself, or the block that it stands in
        own = re.split(r"[;{}]", epilogue[:m.start()])[-1]
        around = " ".join(_headers(epilogue, m.start()))
        assert "!dry" in own or "!dry" in around or "dry ? BN" in around, m.group()
    parts = gemm[gemm.index("struct Epilogue {"):gemm.index("void gemm_body(")]
    send = parts[parts.index("void send("):]
    assert send.index("if (rehearsing()) return;") < send.index("tma_store_3d(")
    gated = parts[parts.index("bool gated_tile("):]
    assert "ch < (rehearsing() ? 1 : BN / CHUNK)" in gated and "!rehearsing() && !mbar_wait_warp(" in gated
    at = gated.index("request(")
    assert _headers(gated, at)[0].startswith("if (ch > 0 &&") and "request(" not in gated[:at]     # not in the first chunk's round
    assert "norm_heads > 0 && !rehearsing();" in parts and re.search(r"if \(more\) load_angles\(", parts)
    # the attention's rows of that round lie past the end, its flags are dropped
    attn = _code("attention.cu")
    assert "const Item it = i < 0 ? Item{(p.rows + BM - 1) / BM * BM, 0, 0} : item_at(i);" in attn
    assert "if (flag && i >= 0) {" in attn


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
