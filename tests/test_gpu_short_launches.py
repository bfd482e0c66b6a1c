"""Forms that only the short launches of a plan take: the FFN2 product with its K divided over a cluster, the attention that
rehearses, the launches that open a call."""
import numpy as np
import pytest
import torch

from paper_2607_11136_b200 import binding as xb
from paper_2607_11136_b200.session import BlockSession
from xema_inputs import Template, make_activations, make_block_weights

from gpu_util import assert_bf16_close, from_dev_bf16

pytestmark = pytest.mark.gpu


def _template(batch, tokens, hidden, ffn, heads=None):
    heads = heads or hidden // 64
    return Template("short", batch, 8, 1, 1, tokens - 8, hidden, heads, hidden // heads, ffn)


# (batch, tokens, hidden, ffn, CTAs that share K): few rows, both sides of the 128-row tiles, several batch elements, K blocks
# fewer and more than the stages (8 to 32 a CTA), the most tiles that still share
@pytest.mark.parametrize("batch,tokens,hidden,ffn,split", [
    (1, 9, 512, 2048, 4), (1, 128, 512, 2304, 4), (1, 129, 1024, 4096, 4), (2, 255, 512, 4096, 4), (1, 512, 1024, 4096, 4),
    (1, 577, 1024, 4096, 2), (3, 200, 1024, 4352, 2)])
def test_ffn2_with_k_divided_over_a_cluster(batch, tokens, hidden, ffn, split):
    t = _template(batch, tokens, hidden, ffn)
    w = make_block_weights(t, 3)
    x, temb = make_activations(t)
    outs = []
    for chunks in ((1, 1, 1), (1, 1, min(3, tokens))):
        s = BlockSession(t, [w], chunks=chunks)
        s.set_inputs(x, temb)
        s.forward()
        outs.append(s.output_bits().copy())
        s.check_status()
        if chunks[2] > 1:
            continue
        # the operands of FFN2 outlive it in the arena
        g = s.view("g0_0", torch.int16, (batch, tokens, ffn))
        res = s.view("res0", torch.float32, (batch, tokens, hidden))
        gate = s.view("mod0", torch.float32, (batch, 6 * hidden))[:, 5 * hidden:]
        w2, b2 = s.weights[0]["w_2"], s.weights[0]["b_2"]
        f64 = lambda v: torch.from_numpy(from_dev_bf16(v))
        want = res.double().cpu() + gate.double().cpu()[:, None] * (f64(g) @ f64(w2).T + f64(b2))
        # partial sums add fp32 roundings only: the bound of every other form of the product
        assert_bf16_close(from_dev_bf16(s.hid_out()), want.numpy(), (batch, tokens, hidden, ffn))
        # the undivided sum differs in its last bits, and in a bf16 rounding here and there
        out = torch.empty_like(s.hid_out())
        kw = dict(a=g.data_ptr(), lda=ffn, a_batch_rows=tokens, w=w2.data_ptr(), ldw=ffn, bias=b2.data_ptr(), out=out.data_ptr(),
                  ldo=hidden, out_batch_rows=tokens, resid=res.data_ptr(), ldr=hidden, resid_batch_rows=tokens,
                  gate=gate.data_ptr(), gate_stride=6 * hidden, batch=batch, rows=tokens, N=hidden, K=ffn,
                  epilogue=xb.EPI_GATE_RES_BF16)
        xb.xema_op_gemm(status=s.status.data_ptr(), stream=torch.cuda.current_stream().cuda_stream, **kw)
        tiles = batch * -(-tokens // 128) * (hidden // 128)
        assert tiles * split <= 148 * 7 // 8 and (split == 4 or tiles * 4 > 148 * 7 // 8)
        if tokens > 100:
            assert not torch.equal(out, s.hid_out())
        assert_bf16_close(from_dev_bf16(out), want.numpy(), "undivided")
    assert np.array_equal(outs[0], outs[1])


def test_a_template_of_many_rows_is_not_divided():
    t = _template(1, 1100, 512, 2048)      # 36 tiles of 128 x 128: its FFN2 keeps the bits of xema_op_gemm
    s = BlockSession(t, [make_block_weights(t, 3)], chunks=(1, 1, 1))
    s.set_inputs(*make_activations(t))
    s.forward()
    g, res = s.view("g0_0", torch.int16, (1, 1100, 2048)), s.view("res0", torch.float32, (1, 1100, 512))
    gate = s.view("mod0", torch.float32, (1, 3072))[:, 2560:]
    out = torch.empty_like(s.hid_out())
    xb.xema_op_gemm(status=s.status.data_ptr(), stream=torch.cuda.current_stream().cuda_stream, a=g.data_ptr(), lda=2048,
                    a_batch_rows=1100, w=s.weights[0]["w_2"].data_ptr(), ldw=2048, bias=s.weights[0]["b_2"].data_ptr(),
                    out=out.data_ptr(), ldo=512, out_batch_rows=1100, resid=res.data_ptr(), ldr=512, resid_batch_rows=1100,
                    gate=gate.data_ptr(), gate_stride=3072, batch=1, rows=1100, N=512, K=2048, epilogue=xb.EPI_GATE_RES_BF16)
    assert torch.equal(out, s.hid_out())


# the attention of a plan follows another launch and, up to 8 key blocks a CTA, rehearses; the same call by itself does not
@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("tokens,chunks", [(9, 1), (130, 1), (161, 3), (333, 2), (1024, 1), (1030, 1)])
def test_attention_behind_another_launch_keeps_its_bits(head_dim, tokens, chunks):
    t = _template(1, tokens, 512, 512, heads=512 // head_dim)
    s = BlockSession(t, [make_block_weights(t, 5)], chunks=(1, chunks, 1))
    s.set_inputs(*make_activations(t))
    stream = torch.cuda.current_stream().cuda_stream
    s.plan.forward_prefix(8, stream)       # MOD, LN1A, KV, KROPE, LN1B, Q, QROPE, ATTN of the first chunk
    rows = tokens // chunks
    q, kv = s.view("q0_0", torch.int16, (1, rows, 512)), s.view("kv0", torch.int16, (1, tokens, 1024))
    got = s.view("o0_0", torch.int16, (1, rows, 512)).clone()
    lse = s.view("lse0_0", torch.float32, (1, 512 // head_dim, rows)).clone()
    o, l = torch.empty_like(got), torch.empty_like(lse)
    xb.xema_op_attention(q.data_ptr(), 512, rows, kv.data_ptr(), kv.data_ptr() + 1024, 1024, tokens, o.data_ptr(), l.data_ptr(),
                         1, rows, tokens, 512 // head_dim, head_dim, status=s.status.data_ptr(), stream=stream, q_scale=1.0)
    s.check_status()
    assert torch.equal(o, got) and torch.equal(l, lse)



@pytest.mark.parametrize("tokens", [130, 1030])
def test_calls_back_to_back_see_their_own_inputs_and_weights(tokens):
    """The first launches of a call may start while the work ahead of them runs: inputs, and weights that a kernel of the
    caller writes right before the call, are read only when it has finished."""
    t = _template(1, tokens, 512, 2048)
    ws = [make_block_weights(t, seed) for seed in (1, 2)]
    ins = [make_activations(t, seed) for seed in (3, 4)]
    want = []
    for w, (x, temb) in zip(ws, ins):
        s = BlockSession(t, [w], chunks=(1, 1, 1))
        s.set_inputs(x, temb)
        s.forward()
        want.append(s.output_bits().copy())
    dev = [{k: torch.from_numpy(v.view(np.int16)).cuda() for k, v in w.items()} for w in ws]
    src = [[torch.from_numpy(v.view(np.int16)).cuda() for v in pair] for pair in ins]
    s = BlockSession(t, [{k: v.clone() for k, v in dev[0].items()}], chunks=(1, 1, 1))
    outs = []
    for i in (0, 1, 1, 0, 1, 0):
        x, temb = (v.clone() for v in src[i])
        s.set_inputs(x, temb, non_blocking=True)
        for k, v in s.weights[0].items():
            v.copy_(dev[i][k])
        s.forward()
        outs.append((i, s.hid_out().clone()))
    for i, y in outs:
        assert np.array_equal(y.cpu().numpy().view(np.uint16), want[i].reshape(y.shape))
