"""What the short launches of a plan do differently, and what they must not: the bits of their products, the attention that
rehearses, the launches that open a call."""
import re

import numpy as np
import pytest
import torch

from paper_2607_11136_b200 import binding as xb
from paper_2607_11136_b200.session import BlockSession
from xema_inputs import Template, make_activations, make_block_weights

pytestmark = pytest.mark.gpu


def _template(batch, tokens, hidden, ffn, heads=None):
    heads = heads or hidden // 64
    return Template("short", batch, 8, 1, 1, tokens - 8, hidden, heads, hidden // heads, ffn)


def _op_gemm(s, tokens, N, K, a, w, bias, resid, gate, epilogue):
    """The gated product of a plan of whole phases once more, as the stand-alone operator computes it."""
    t = s.template
    out = torch.empty((t.batch, tokens, N), dtype=torch.float32 if epilogue == xb.EPI_GATE_RES_F32 else torch.int16, device="cuda")
    xb.xema_op_gemm(a=a.data_ptr(), lda=K, a_batch_rows=tokens, w=w.data_ptr(), ldw=K, bias=bias.data_ptr(), out=out.data_ptr(),
                    ldo=N, out_batch_rows=tokens, resid=resid.data_ptr(), ldr=N, resid_batch_rows=tokens, gate=gate.data_ptr(),
                    gate_stride=6 * N, batch=t.batch, rows=tokens, N=N, K=K, epilogue=epilogue, status=s.status.data_ptr(),
                    stream=torch.cuda.current_stream().cuda_stream)
    return out


# few rows, widths and K that leave SMs without a tile: one sum over K in order, whatever the plan
@pytest.mark.parametrize("batch,tokens,hidden,ffn", [
    (1, 9, 512, 2048), (1, 128, 512, 2304), (1, 129, 1024, 4096), (2, 255, 512, 4096), (1, 333, 1024, 4096), (1, 577, 1024, 4096),
    (3, 200, 1024, 4352), (1, 256, 2048, 2048), (2, 120, 1536, 1536), (1, 100, 3072, 3072), (1, 1100, 512, 2048)])
def test_gated_products_of_a_plan_have_the_bits_of_the_operator(batch, tokens, hidden, ffn):
    s = BlockSession(_template(batch, tokens, hidden, ffn), [make_block_weights(_template(batch, tokens, hidden, ffn), 3)],
                     chunks=(1, 1, 1))
    s.set_inputs(*make_activations(s.template))
    w, rows = s.weights[0], (batch, tokens)
    mod = s.view("mod0", torch.float32, (batch, 6 * hidden))
    s.plan.forward_prefix(9, torch.cuda.current_stream().cuda_stream)      # up to PROJ
    res = s.view("res0", torch.float32, rows + (hidden,))
    proj = _op_gemm(s, tokens, hidden, hidden, s.view("o0_0", torch.int16, rows + (hidden,)), w["w_o"], w["b_o"],
                    s.view("hid0", torch.int16, rows + (hidden,)), mod[:, 2 * hidden:], xb.EPI_GATE_RES_F32)
    assert torch.equal(proj, res)
    s.forward()                            # (the operands of FFN2 outlive it in the arena)
    ffn2 = _op_gemm(s, tokens, hidden, ffn, s.view("g0_0", torch.int16, rows + (ffn,)), w["w_2"], w["b_2"], res,
                    mod[:, 5 * hidden:], xb.EPI_GATE_RES_BF16)
    assert torch.equal(ffn2, s.hid_out())
    s.check_status()


@pytest.mark.parametrize("tokens,hidden", [(200, 512), (333, 1024)])
def test_a_request_has_the_same_bits_alone_and_in_a_batch(tokens, hidden):
    t = _template(3, tokens, hidden, 4 * hidden)
    w = make_block_weights(t, 3)
    x, temb = make_activations(t)
    outs = []
    for first, n in ((0, 3), (0, 1), (1, 2), (2, 1)):
        s = BlockSession(_template(n, tokens, hidden, 4 * hidden), [w], chunks=(1, 1, 1))
        s.set_inputs(np.ascontiguousarray(x[first:first + n]), np.ascontiguousarray(temb[first:first + n]))
        s.forward()
        outs.append((first, n, s.output_bits().copy()))
        s.check_status()
    for first, n, y in outs[1:]:
        assert np.array_equal(y, outs[0][2][first:first + n]), (first, n)


# One tile form after the other: single 64, pair 128 and pair 256, rows at and beside their edges, both head sizes, a shard.
@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("batch,hidden,tokens,shard", [
    (1, 512, 9, None), (1, 512, 128, None), (2, 512, 129, None), (3, 1024, 200, None), (1, 1536, 1025, None), (1, 2048, 1280, None),
    (1, 3072, 2561, None), (1, 512, 300, (1, 2))])
def test_keys_values_and_queries_in_one_launch_have_the_bits_of_two(head_dim, batch, hidden, tokens, shard):
    t = _template(batch, tokens, hidden, 512, heads=hidden // head_dim)
    s = BlockSession(t, [make_block_weights(t, 7)], chunks=(1, 1, 1), shard=shard)
    assert s.plan.forward_launches() == s.plan.launch_count() - 1
    x, temb = make_activations(t)
    r0, rows = (0, tokens) if shard is None else (s.plan.row0, s.plan.rows)
    stream = torch.cuda.current_stream().cuda_stream
    got = []
    for ends in (range(1, 8), [7]):              # MOD, LN1A, KV, KROPE, LN1B, Q, QROPE one by one, and in one call
        s.arena.fill_(0x5A)
        s.set_inputs(np.ascontiguousarray(x[:, r0:r0 + rows]), temb)
        for first, end in zip([0] + list(ends), ends):
            s.plan.forward_range(first, end, stream)
        got.append((s.view("q0_0", torch.int16, (batch, rows, hidden)).clone(),
                    s.view("kv0", torch.int16, (batch, tokens, 2 * hidden)).clone()))
        s.check_status()
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


# One and several batch elements, whole and cut phases, a width without an instance that carries a modulation, a shard.
@pytest.mark.parametrize("batch,hidden,tokens,chunks,shard,carried", [
    (1, 512, 9, (1, 1, 1), None, 2), (3, 768, 130, (1, 1, 1), None, 2), (5, 512, 33, (2, 1, 3), None, 2), (1, 3072, 40, (1, 2, 2), None, 2),
    (1, 3328, 40, (1, 1, 1), None, 0), (2, 512, 100, (1, 1, 1), (1, 2), 2)])
def test_a_step_has_the_same_bits_wherever_it_is_cut(batch, hidden, tokens, chunks, shard, carried):
    """Launches that take a neighbouring operator along (Q beside KV, a later block's modulation beside LN2 and LN1A) do so only
    where the call covers all that is involved."""
    t = _template(batch, tokens, hidden, 512)
    t = Template(t.name, *[getattr(t, f) for f in ("batch", "s_text", "grid_t", "grid_h", "grid_w", "hidden", "heads", "head_dim", "ffn")],
                 n_blocks=3)
    s = BlockSession(t, [make_block_weights(t, seed) for seed in range(3)], chunks=chunks, shard=shard)
    joint = 3 if chunks[:2] == (1, 1) else 0
    assert s.plan.forward_launches() == s.plan.launch_count() - joint - carried
    x, temb = make_activations(t)
    r0, rows = (0, tokens) if shard is None else (s.plan.row0, s.plan.rows)
    x = torch.from_numpy(np.ascontiguousarray(x[:, r0:r0 + rows]).view(np.int16)).cuda()
    temb = torch.from_numpy(temb.view(np.int16)).cuda()
    n, stream = s.plan.n_ops, torch.cuda.current_stream().cuda_stream
    outs = []
    for cuts in [range(1, n)] + [[]] + [[c] for c in range(1, n)]:
        s.arena.fill_(0)             # (a shard's missing keys)
        s.set_inputs(x, temb)
        for first, end in zip([0] + list(cuts), list(cuts) + [n]):
            s.plan.forward_range(first, end, stream)
        outs.append(s.hid_out().clone())
    s.check_status()
    assert len(outs) == n + 1 and outs[0].any()
    for cut, y in enumerate(outs[1:]):
        assert torch.equal(y, outs[0]), cut


# Both sides of every line of the rule; a launch that carries, and one of many rows, has the bits of the launches apart.
@pytest.mark.parametrize("batch,hidden,tokens,carried", [
    (1, 512, 4096, 1), (1, 512, 4097, 0), (1, 3072, 300, 1), (1, 3328, 300, 0), (2, 512, 2048, 1), (2, 512, 2049, 0), (2, 2816, 65, 1),
    (4, 512, 24, 1), (4, 512, 100, 0), (4, 512, 200, 1), (4, 512, 513, 0), (5, 512, 200, 0), (3, 1024, 682, 1), (3, 1024, 683, 0),
    (4, 1280, 256, 1), (4, 1280, 257, 0), (6, 2048, 85, 1), (6, 2048, 86, 0), (3, 2304, 20, 0), (7, 1024, 40, 0), (1, 512, 8193, 0)])
def test_a_modulation_is_carried_where_that_is_faster(batch, hidden, tokens, carried):
    t = _template(batch, tokens, hidden, 256)
    t = Template(t.name, *[getattr(t, f) for f in ("batch", "s_text", "grid_t", "grid_h", "grid_w", "hidden", "heads", "head_dim", "ffn")],
                 n_blocks=2)
    w = [make_block_weights(t, 1), make_block_weights(t, 2)]
    s = BlockSession(t, w, chunks=(1, 1, 1))
    assert s.plan.forward_launches() == s.plan.launch_count() - 2 - carried       # (both blocks' Q goes with KV)
    x, temb = (torch.from_numpy(a.view(np.int16)).cuda() for a in make_activations(t))
    stream, outs = torch.cuda.current_stream().cuda_stream, []
    for ends in ([s.plan.n_ops], range(1, s.plan.n_ops + 1)):
        s.arena.fill_(0x5A)
        s.set_inputs(x, temb)
        for first, end in zip([0] + list(ends), ends):
            s.plan.forward_range(first, end, stream)
        outs.append(s.hid_out().clone())
    s.check_status()
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("batch,hidden,tokens,chunks", [(1, 512, 200, (1, 1, 1)), (2, 768, 130, (1, 1, 3)), (3, 1024, 77, (1, 1, 1))])
def test_launches_that_take_a_neighbour_along_write_their_results_and_nothing_else(batch, hidden, tokens, chunks):
    """Over an arena with 4 KiB free behind every tensor: the calls that run KV .. Q in one launch and LN2 .. LN1A with the next
    block's modulation inside change bytes of their operators' results only, neither other tensors nor what lies between them."""
    t = _template(batch, tokens, hidden, 512)
    t = Template(t.name, *[getattr(t, f) for f in ("batch", "s_text", "grid_t", "grid_h", "grid_w", "hidden", "heads", "head_dim", "ffn")],
                 n_blocks=3)
    s = BlockSession(t, [make_block_weights(t, seed) for seed in range(3)], chunks=chunks, guard_bytes=4096)
    assert s.plan.forward_launches() == s.plan.launch_count() - 5
    names = [s.plan.op(k)["name"] for k in range(s.plan.n_ops)]
    calls = []                                   # (first op, end, tensors that they write)
    for l, kv in enumerate(k for k, name in enumerate(names) if name == "KV"):
        assert names[kv:kv + 4] == ["KV", "KROPE", "LN1B", "Q"]
        calls.append((kv, kv + 4, ["kv%d" % l, "q%d_0" % l]))
    for l, mod in enumerate((k for k, name in enumerate(names) if name == "MOD" and k), start=1):
        assert names[mod - 3:mod + 2] == ["LN2", "FFN1", "FFN2", "MOD", "LN1A"]
        last = chunks[2] - 1
        calls.append((mod - 3, mod + 2, ["h2%d_%d" % (l - 1, last), "g%d_%d" % (l - 1, last), "hid%d" % l, "mod%d" % l, "h1a%d_0" % l]))
    stream, at = torch.cuda.current_stream().cuda_stream, 0
    s.arena.fill_(0xA5)
    s.set_inputs(*make_activations(t))
    for first, end, written in sorted(calls):
        s.plan.forward_range(at, first, stream)
        before = s.arena.clone()
        s.plan.forward_range(first, end, stream)
        changed = s.arena != before
        for name in written:
            off, nbytes = s.plan.tensor(name)
            assert changed[off:off + nbytes].any(), (first, name)
        for name in written:
            off, nbytes = s.plan.tensor(name)
            changed[off:off + nbytes] = False
        assert not changed.any(), (first, changed.nonzero()[:4].tolist())
        at = end
    s.check_status()


def _attention_of_a_plan(batch, heads, head_dim, tokens, chunks):
    """A session that has run up to its first attention launch: MOD, LN1A, KV, KROPE, LN1B, Q, QROPE, ATTN."""
    t = _template(batch, tokens, heads * head_dim, 512, heads=heads)
    s = BlockSession(t, [make_block_weights(t, 5)], chunks=(1, chunks, 1))
    s.set_inputs(*make_activations(t))
    s.plan.forward_prefix(8, torch.cuda.current_stream().cuda_stream)
    return s


# The attention of a plan follows another launch and, up to 8 key blocks a CTA, rehearses; the same call by itself does not.
# One tile per item and two, one item per CTA and two, up to 8 key blocks and beyond.
@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("batch,hidden,tokens,chunks", [
    (1, 512, 9, 1), (1, 512, 130, 1), (1, 512, 161, 3), (1, 512, 333, 2), (1, 512, 1024, 1), (1, 512, 1030, 1),
    (4, 1536, 257, 1), (8, 1536, 257, 1), (8, 1536, 400, 1), (8, 1536, 500, 4)])
def test_attention_behind_another_launch_keeps_its_bits(head_dim, batch, hidden, tokens, chunks):
    heads = hidden // head_dim
    s = _attention_of_a_plan(batch, heads, head_dim, tokens, chunks)
    rows = tokens // chunks
    q, kv = s.view("q0_0", torch.int16, (batch, rows, hidden)), s.view("kv0", torch.int16, (batch, tokens, 2 * hidden))
    got = s.view("o0_0", torch.int16, (batch, rows, hidden)).clone()
    lse = s.view("lse0_0", torch.float32, (batch, heads, rows)).clone()
    o, l = torch.empty_like(got), torch.empty_like(lse)
    xb.xema_op_attention(q.data_ptr(), hidden, rows, kv.data_ptr(), kv.data_ptr() + 2 * hidden, 2 * hidden, tokens, o.data_ptr(),
                         l.data_ptr(), batch, rows, tokens, heads, head_dim, status=s.status.data_ptr(),
                         stream=torch.cuda.current_stream().cuda_stream, q_scale=1.0)
    s.check_status()
    assert torch.equal(o, got) and torch.equal(l, lse)


# (batch 8: 192 items over 148 SMs, whether a head has one row tile or two)
@pytest.mark.parametrize("batch,tokens,chunks,rehearses", [
    (1, 1024, 1, True), (1, 1025, 1, False), (8, 500, 4, True), (8, 600, 5, False), (8, 512, 2, True), (8, 513, 2, False)])
def test_attention_rehearses_up_to_eight_key_blocks_a_cta(batch, tokens, chunks, rehearses):
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA], acc_events=True) as prof:
        _attention_of_a_plan(batch, 24, 64, tokens, chunks)
        torch.cuda.synchronize()
    names = [re.search(r"attention_kernel<([^>]*)>", e.name) for e in prof.events() if "attention_kernel" in e.name]
    assert len(names) == 1
    assert names[0].group(1).split(",")[2].strip().replace("(bool)", "") in (("1", "true") if rehearses else ("0", "false"))


MASK = 0x5a5a


class _Tail:
    """Device tensors at the end of a large buffer.  `write(i)` puts source `i` there with one kernel that works through the whole
    buffer, some 50 us, and comes to the tensors last: what is launched right behind it is there before they are written."""

    def __init__(self, sources):
        shapes = {k: v.shape for k, v in sources[0].items()}
        end = [0]
        for v in sources[0].values():
            assert v.size % 8 == 0               # every tensor starts on a 16-byte boundary
            end.append(end[-1] + v.size)
        lead = (1 << 26) - end[-1]
        self.live = torch.zeros(1 << 26, dtype=torch.int16, device="cuda")
        self.sources = []
        for src in sources:
            flat = torch.from_numpy(np.concatenate([v.reshape(-1) for v in src.values()]).view(np.int16)).cuda()
            self.sources.append(torch.zeros_like(self.live))
            self.sources[-1][lead:] = flat ^ MASK
        self.tensors = {k: self.live[lead + at:lead + at + int(np.prod(shape))].view(shape)
                        for (k, shape), at in zip(shapes.items(), end)}

    def write(self, i):
        torch.bitwise_xor(self.sources[i], MASK, out=self.live)


@pytest.mark.parametrize("tokens", [130, 1030])
def test_calls_see_what_a_kernel_wrote_right_before_them(tokens):
    """The copy of set_inputs is launched while the work ahead of it still runs, and weights are requested ahead of a launch's own
    wait: inputs and weights of a call are those that the caller's last kernel before it wrote, and its output is the
    caller's until the next call.  Nothing but kernels stands between the calls: no copy, no synchronisation."""
    t = _template(1, tokens, 512, 2048)
    ws = [make_block_weights(t, seed) for seed in (1, 2)]
    ins = [dict(zip(("x", "temb"), make_activations(t, seed))) for seed in (3, 4)]
    want = {}
    for i, w in enumerate(ws):
        for j, a in enumerate(ins):
            s = BlockSession(t, [w], chunks=(1, 1, 1))
            s.set_inputs(a["x"], a["temb"])
            s.forward()
            want[i, j] = s.output_bits().copy()
    weights, inputs = _Tail(ws), _Tail(ins)
    ready = [{k: torch.from_numpy(v.view(np.int16)).cuda() for k, v in a.items()} for a in ins]
    s = BlockSession(t, [weights.tensors], chunks=(1, 1, 1))
    outs, got = torch.empty((14,) + s.hid_out().shape, dtype=torch.int16, device="cuda"), []

    def collect(i, j):
        torch.bitwise_xor(s.hid_out(), MASK, out=outs[len(got)])
        got.append((i, j))

    weights.write(0)
    torch.cuda.synchronize()
    for j in (0, 1, 1, 0):                       # inputs written right before set_inputs
        inputs.write(j)
        s.set_inputs(inputs.tensors["x"], inputs.tensors["temb"])
        s.forward()
        collect(0, j)
    for j in (1, 0, 1):                          # nothing between a call and the next one's inputs
        for k in (1 - j, j):
            s.set_inputs(ready[k]["x"], ready[k]["temb"])
            s.forward()
        collect(0, j)
    for i in (1, 0, 0, 1):                       # weights written right before forward
        s.set_inputs(ready[0]["x"], ready[0]["temb"])
        weights.write(i)
        s.forward()
        collect(i, 0)
    for i in (0, 1, 0):                          # weights written right before set_inputs
        weights.write(i)
        s.set_inputs(ready[1]["x"], ready[1]["temb"])
        s.forward()
        collect(i, 1)
    s.check_status()
    for (i, j), y in zip(got, outs):
        assert np.array_equal((y ^ MASK).cpu().numpy().view(np.uint16), want[i, j].reshape(y.shape)), (i, j)


# rows of several waves of tiles; the output over h2 of the first chunk, four rows behind it and apart from it; batch elements
@pytest.mark.parametrize("batch,tokens,hidden,chunks,over", [
    (1, 6930, 3072, (1, 1, 1), "at"), (1, 13000, 3072, (1, 1, 2), "at"), (1, 17776, 3072, (1, 1, 3), "behind"), (3, 2500, 2048, (1, 1, 1), "at"),
    (2, 4800, 1536, (1, 1, 2), "at")])
def test_forward_host_cuts_the_first_feed_forward_chunk(batch, tokens, hidden, chunks, over):
    t = _template(batch, tokens, hidden, 12288 if over == "behind" else 1024)
    s = BlockSession(t, [make_block_weights(t, 2)], chunks=chunks)
    (out, _), (h2, _) = s.plan.tensor("hid1"), s.plan.tensor("h20_0")
    assert (out == h2) == (over == "at") and (out > h2) == (over == "behind")
    x, temb = (torch.from_numpy(a.view(np.int16)) for a in make_activations(t))
    s.set_inputs(x, temb)
    s.forward()
    want = s.hid_out().cpu()
    x, temb = x.pin_memory(), temb.pin_memory()
    y = torch.empty_like(x).pin_memory()
    for fill in (0xFF, 0x00):
        s.arena.fill_(fill)
        s.plan.forward_host(x.data_ptr(), temb.data_ptr(), y.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        s.check_status()
        assert torch.equal(y, want), fill


# LN2 launches of the call: of a first chunk that is cut and, where a piece of the output would end behind h2's rows that are still to
# come, of one that is not (the output four rows behind h2; two row chunks of three batch elements)
@pytest.mark.parametrize("batch,tokens,hidden,ffn,chunks,launches", [
    (1, 6930, 3072, 1024, (1, 1, 1), [4]), (1, 17776, 3072, 12288, (1, 1, 3), [1, 4, 4]), (2, 4800, 1536, 1024, (1, 1, 2), [2, 2]),
    (3, 3200, 1536, 1024, (1, 1, 2), [1, 3])])
def test_forward_host_leaves_a_first_chunk_whole_where_its_pieces_would_meet(batch, tokens, hidden, ffn, chunks, launches):
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the pieces are counted for 148 SMs")
    t = _template(batch, tokens, hidden, ffn)
    s = BlockSession(t, [make_block_weights(t, 2)], chunks=chunks)
    x, temb = (torch.from_numpy(a.view(np.int16)) for a in make_activations(t))
    s.set_inputs(x, temb)
    s.forward()
    want = s.hid_out().cpu()
    x, temb = x.pin_memory(), temb.pin_memory()
    y = torch.empty_like(x).pin_memory()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA], acc_events=True) as prof:
        s.plan.forward_host(x.data_ptr(), temb.data_ptr(), y.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
    s.check_status()
    assert torch.equal(y, want)
    ln2 = [e for e in prof.events() if re.search(r"ln_modulate_kernel<(\(bool\))?(1|true),", e.name)]     # (float32 rows)
    assert len(ln2) == sum(launches)
