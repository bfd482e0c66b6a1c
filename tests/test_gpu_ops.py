"""Per-kernel parity against the oracle's operator definitions, through the C ABI (GPU)."""
import json
import math

import numpy as np
import pytest
import torch

from oracle import block as ob
from paper_2607_11136_b200 import binding as xb
from xema_inputs import bf16_bits, bits_to_f64, template

from gpu_util import DEV, assert_bf16_close, assert_close, from_dev_bf16, rand_bf16, to_dev

pytestmark = pytest.mark.gpu


def _sync_status(status):
    torch.cuda.synchronize()
    assert int(status.item()) == 0, "device status 0x%08x" % (int(status.item()) & 0xFFFFFFFF)


def test_mod_gemv():
    rng = np.random.default_rng(0)
    for B, Dt, n_out in ((1, 512, 3072), (4, 512, 6 * 3072), (3, 64, 40)):
        tb, tf = rand_bf16(rng, (B, Dt))
        wb, wf = rand_bf16(rng, (n_out, Dt), 0.02)
        bb, bf = rand_bf16(rng, (n_out,), 0.02)
        out = torch.empty(B, n_out, dtype=torch.float32, device=DEV)
        t_dev, w_dev, b_dev = to_dev(tb), to_dev(wb), to_dev(bb)
        xb.xema_op_mod(t_dev.data_ptr(), w_dev.data_ptr(), b_dev.data_ptr(), out.data_ptr(), B, Dt, n_out)
        torch.cuda.synchronize()
        ref = ob.linear(ob.silu(tf), wf, bf)
        assert_close(out.cpu().numpy(), ref, "mod", rel=1e-4, cos=0.999999)


# one element and several (a pass takes four), features and inputs beside the warps' and lanes' shares, an odd address
@pytest.mark.parametrize("B,Dt,n_out,shift", [(1, 512, 1, 0), (1, 8, 33, 0), (1, 1032, 257, 1), (2, 520, 31, 1), (4, 512, 64, 0), (5, 1032, 130, 3)])
def test_mod_gemv_edges(B, Dt, n_out, shift):
    rng = np.random.default_rng(B * Dt + n_out)
    tb, tf = rand_bf16(rng, (B, Dt))
    wb, wf = rand_bf16(rng, (n_out, Dt), 0.02)
    bb, bf = rand_bf16(rng, (n_out,), 0.02)
    out = torch.full((B * n_out + 1,), 7.0, dtype=torch.float32, device=DEV)
    room = torch.empty(B * Dt + shift, dtype=torch.int16, device=DEV)
    room[shift:] = to_dev(tb).reshape(-1)
    w_dev, b_dev = to_dev(wb), to_dev(bb)
    xb.xema_op_mod(room.data_ptr() + 2 * shift, w_dev.data_ptr(), b_dev.data_ptr(), out.data_ptr(), B, Dt, n_out)
    torch.cuda.synchronize()
    ref = ob.linear(ob.silu(tf), wf, bf)
    assert_close(out[:-1].view(B, n_out).cpu().numpy(), ref, "mod", rel=1e-4, cos=0.999999)
    assert out[-1].item() == 7.0


# scale and shift on a 32-byte boundary in every row, in the first only, and in none; widths with a row in registers and beyond
@pytest.mark.parametrize("D", [256, 2048, 2816, 3072, 4352])
def test_ln_modulate_wide_loads_change_nothing(D):
    gen = torch.Generator(device=DEV).manual_seed(D)
    B, rows = 2, 37
    x = torch.randn(B, rows, D, device=DEV, generator=gen).to(torch.bfloat16)
    vals = torch.randn(B, 2, D, device=DEV, generator=gen)
    outs = []
    for first, stride in ((0, 2 * D), (0, 2 * D + 4), (4, 2 * D)):
        mod = torch.zeros(first + 2 * stride + 2 * D, device=DEV)
        for b in range(B):
            mod[first + b * stride:first + b * stride + 2 * D] = vals[b].reshape(-1)
        out = torch.empty(B, rows, D, dtype=torch.bfloat16, device=DEV)
        at = mod.data_ptr() + 4 * first
        xb.xema_op_ln_modulate(x.data_ptr(), 0, rows, out.data_ptr(), at, at + 4 * D, stride, B, rows, D, 1e-6)
        outs.append(out)
    f = x.double()
    f = (f - f.mean(-1, keepdim=True)) / torch.sqrt(f.var(-1, unbiased=False, keepdim=True) + 1e-6)
    want = f * (1 + vals[:, 1:2].double()) + vals[:, :1].double()
    assert_bf16_close(outs[0].double().cpu().numpy(), want.cpu().numpy(), "LN")
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


# Every width whose rows stay in registers: four blocks of 128 threads an SM up to 3072 columns, three up to 4096, in 65536 registers.
def test_ln_modulate_leaves_room_for_other_blocks(tmp_path):
    widths, rows = range(256, 4097, 256), 5
    gen = torch.Generator(device=DEV).manual_seed(7)
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA], acc_events=True) as prof:
        for D in widths:
            x = torch.randn(rows, D, device=DEV, generator=gen).to(torch.bfloat16)
            mod = torch.randn(2, D, device=DEV, generator=gen)
            out = torch.empty_like(x)
            xb.xema_op_ln_modulate(x.data_ptr(), 0, rows, out.data_ptr(), mod.data_ptr(), mod.data_ptr() + 4 * D, 0, 1, rows, D, 1e-6)
            f = x.double()
            f = (f - f.mean(-1, keepdim=True)) / torch.sqrt(f.var(-1, unbiased=False, keepdim=True) + 1e-6)
            assert_bf16_close(out.double().cpu().numpy(), (f * (1 + mod[1].double()) + mod[0].double()).cpu().numpy(), "LN %d" % D)
        torch.cuda.synchronize()
    prof.export_chrome_trace(str(tmp_path / "trace.json"))
    events = [e for e in json.load(open(tmp_path / "trace.json"))["traceEvents"] if "ln_modulate_kernel" in e.get("name", "")]
    assert len(events) == len(widths)
    for D, e in zip(widths, sorted(events, key=lambda e: e["ts"])):
        assert e["args"]["registers per thread"] <= (128 if D <= 3072 else 168), (D, e["args"])


@pytest.mark.parametrize("D,in_f32", [(512, 0), (512, 1), (3072, 0), (3072, 1), (768, 0), (1280, 1)])
def test_ln_modulate(D, in_f32):
    rng = np.random.default_rng(1)
    B, S, rows, row0 = 2, 70, 37, 11
    if in_f32:
        xf32 = (rng.standard_normal((B, S, D), dtype=np.float32) * 1.5 + 0.3).astype(np.float32)
        x_dev, xf = torch.from_numpy(xf32).to(DEV), xf32.astype(np.float64)
        base = x_dev.data_ptr() + row0 * D * 4
    else:
        xbits, xf = rand_bf16(rng, (B, S, D), 1.5)
        x_dev = to_dev(xbits)
        base = x_dev.data_ptr() + row0 * D * 2
    mod = rng.standard_normal((B, 6 * D), dtype=np.float32) * 0.3
    mod_dev = torch.from_numpy(mod).to(DEV)
    out = torch.empty(B, rows, D, dtype=torch.int16, device=DEV)
    xb.xema_op_ln_modulate(base, in_f32, S, out.data_ptr(), mod_dev.data_ptr(), mod_dev.data_ptr() + D * 4, 6 * D, B,
                           rows, D, 1e-6)
    torch.cuda.synchronize()
    m64 = mod.astype(np.float64)
    ref = ob.layer_norm(xf[:, row0:row0 + rows], 1e-6) * (1 + m64[:, None, D:2 * D]) + m64[:, None, :D]
    assert_bf16_close(from_dev_bf16(out), ref, "ln", atol_rms=1e-4)


@pytest.mark.parametrize("D", [256, 1024, 2304, 4096, 4352])
@pytest.mark.parametrize("rows", [1, 3, 5])
def test_ln_modulate_widths(D, rows):
    """Every kind of row the kernel has an instance for: one step per lane, odd step counts, the
    widest row kept in registers and one beyond it, with rows that do not fill a block's warps.
    The result is rounded to bf16 once; 1e-4 of RMS covers the fp32 sums over D terms."""
    rng = np.random.default_rng(5 + D)
    B = 2
    for in_f32 in (0, 1):
        xf32 = (rng.standard_normal((B, rows, D), dtype=np.float32) * 2 + 0.5).astype(np.float32)
        bits = bf16_bits(xf32)
        x_dev = torch.from_numpy(xf32).to(DEV) if in_f32 else to_dev(bits)
        xf = xf32.astype(np.float64) if in_f32 else bits_to_f64(bits)
        mod = rng.standard_normal((B, 2 * D), dtype=np.float32) * 0.3
        mod_dev = torch.from_numpy(mod).to(DEV)
        out = torch.empty(B, rows, D, dtype=torch.int16, device=DEV)
        xb.xema_op_ln_modulate(x_dev.data_ptr(), in_f32, rows, out.data_ptr(), mod_dev.data_ptr(),
                               mod_dev.data_ptr() + D * 4, 2 * D, B, rows, D, 1e-6)
        torch.cuda.synchronize()
        m64 = mod.astype(np.float64)
        ref = ob.layer_norm(xf, 1e-6) * (1 + m64[:, None, D:]) + m64[:, None, :D]
        assert_bf16_close(from_dev_bf16(out), ref, ("ln widths", D, rows, in_f32), atol_rms=1e-4)


@pytest.mark.parametrize("name", ["tiny", "flux"])
def test_rmsnorm_rope(name):
    t = template(name)
    rng = np.random.default_rng(2)
    B, H, dh = 2, 6, t.head_dim
    S = t.seq
    rows, pos0 = 45, t.s_text - 7                     # spans the text / video boundary
    ld = 2 * H * dh + 8 * 3                           # strided rows, like the K half of kv
    xbits, xf = rand_bf16(rng, (B, S, ld), 2.0)
    gb, gf = rand_bf16(rng, (dh,), 1.0)
    x_dev, g_dev = to_dev(xbits), to_dev(gb)
    rope = torch.from_numpy(xb.xema_rope_table(xb.make_config(t))).to(DEV)
    xb.xema_op_rmsnorm_rope(x_dev.data_ptr() + pos0 * ld * 2, ld, S, g_dev.data_ptr(), rope.data_ptr(), pos0, B,
                            rows, H, dh, 1e-6)
    torch.cuda.synchronize()
    got = from_dev_bf16(x_dev)
    ang = ob.rope_angles(t)[pos0:pos0 + rows]
    ref = xf.copy()
    for b in range(B):
        v = xf[b, pos0:pos0 + rows, :H * dh].reshape(rows, H, dh)
        ref[b, pos0:pos0 + rows, :H * dh] = ob.apply_rope(ob.rms_norm(v, gf, 1e-6), ang).reshape(rows, H * dh)
    # untouched: other rows, and the features beyond heads*dh of the touched rows
    mask = np.ones_like(ref, bool)
    mask[:, pos0:pos0 + rows, :H * dh] = False
    assert np.array_equal(got[mask], xf[mask])
    assert_bf16_close(got[~mask], ref[~mask], "rmsnorm_rope", atol_rms=1e-4)


def _gemm_case(rng, B, rows, N, K, epi, a_extra_rows=5, tile=None):
    ab, af = rand_bf16(rng, (B, rows + a_extra_rows, K))
    wb, wf = rand_bf16(rng, (N, K), 0.05)
    bb, bf = rand_bf16(rng, (N,), 0.5)
    a_dev, w_dev, b_dev = to_dev(ab), to_dev(wb), to_dev(bb)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    out_rows = rows + 3                                 # output lives inside a larger tensor
    acc = af[:, :rows] @ wf.T + bf
    kw = dict(a=a_dev.data_ptr(), lda=K, a_batch_rows=rows + a_extra_rows, w=w_dev.data_ptr(), ldw=K,
              bias=b_dev.data_ptr(), ldo=N, out_batch_rows=out_rows, batch=B, rows=rows, N=N, K=K, epilogue=epi)
    keep = [a_dev, w_dev, b_dev]
    if epi in (xb.EPI_BIAS, xb.EPI_BIAS_GELU):
        out = torch.full((B, out_rows, N), 0x7FC0, dtype=torch.int16, device=DEV)
        ref = acc if epi == xb.EPI_BIAS else ob.gelu_tanh(acc)
    else:
        gate = rng.standard_normal((B, N), dtype=np.float32) * 0.3
        g_dev = torch.from_numpy(gate).to(DEV)
        keep.append(g_dev)
        kw.update(gate=g_dev.data_ptr(), gate_stride=N, ldr=N, resid_batch_rows=rows)
        if epi == xb.EPI_GATE_RES_F32:
            rb, rf = rand_bf16(rng, (B, rows, N))
            r_dev = to_dev(rb)
            out = torch.full((B, out_rows, N), float("nan"), dtype=torch.float32, device=DEV)
        else:
            r32 = rng.standard_normal((B, rows, N), dtype=np.float32)
            rf, r_dev = r32.astype(np.float64), torch.from_numpy(r32).to(DEV)
            out = torch.full((B, out_rows, N), 0x7FC0, dtype=torch.int16, device=DEV)
        keep.append(r_dev)
        kw.update(resid=r_dev.data_ptr())
        ref = rf + gate.astype(np.float64)[:, None, :] * acc
    kw.update(out=out.data_ptr())
    if tile is None:
        xb.xema_op_gemm(status=status.data_ptr(), **kw)
    else:
        xb.xema_op_gemm_in_tile(*tile, status=status.data_ptr(), **kw)
    _sync_status(status)
    got = out.cpu().numpy().astype(np.float64) if out.dtype == torch.float32 else from_dev_bf16(out)
    # rows past `rows` of every batch element must be untouched
    tail = out[:, rows:].cpu().numpy()
    if out.dtype == torch.float32:
        assert np.isnan(tail).all()
    else:
        assert (tail.view(np.uint16) == 0x7FC0).all()
    return got[:, :rows], ref


@pytest.mark.parametrize("epi", [0, 1, 2, 3])
@pytest.mark.parametrize("B,rows,N,K", [(1, 128, 256, 64), (1, 300, 512, 512), (2, 77, 384, 192),
                                        (1, 1000, 3072, 3072), (1, 129, 1024, 2048), (3, 257, 256, 128),
                                        (1, 5000, 768, 320)])
def test_gemm_epilogues(epi, B, rows, N, K):
    rng = np.random.default_rng(100 + epi)
    got, ref = _gemm_case(rng, B, rows, N, K, epi)
    if epi == xb.EPI_GATE_RES_F32:
        assert_close(got, ref, ("gemm", epi, B, rows, N, K), rel=1e-4, cos=0.9999999)      # fp32 output
    else:
        assert_bf16_close(got, ref, ("gemm", epi, B, rows, N, K), atol_rms=2e-3 if epi == xb.EPI_BIAS_GELU else 2e-4)


@pytest.mark.parametrize("epi", [0, 1, 2, 3])
@pytest.mark.parametrize("rows", [1, 31, 33, 127, 160, 225, 257])
def test_gemm_epilogue_row_edges(epi, rows):
    """Rows that end inside, at and just past a warp's 32 and a tile's 128 / 256 rows, in the tiles that
    problems of this size get (one CTA, 64 or 32 columns; every tile: the next test), two batch
    elements: the results leave in boxes of 32 rows x 32 columns, and rows past the end must stay
    untouched (checked by _gemm_case).  Tolerances as in test_gemm_epilogues: half a bf16 spacing of the output, 1e-4 of
    RMS for fp32 sums of K = 192 products."""
    for N in (384, 512):
        got, ref = _gemm_case(np.random.default_rng(300 + rows + epi), 2, rows, N, 192, epi)
        if epi == xb.EPI_GATE_RES_F32:
            assert_close(got, ref, ("gemm edges", epi, rows, N), rel=1e-4, cos=0.9999999)
        else:
            assert_bf16_close(got, ref, ("gemm edges", epi, rows, N), atol_rms=2e-3 if epi == xb.EPI_BIAS_GELU else 2e-4)


TILES = [(1, 256), (1, 128), (0, 128), (0, 64), (0, 32)]      # (CTA pair, columns)


@pytest.mark.parametrize("epi", [0, 1, 2, 3])
@pytest.mark.parametrize("tile", TILES)
def test_gemm_row_edges_in_every_tile(epi, tile):
    """The same edges with the tile named: warps, and the second CTA of a pair, whose rows lie wholly past
    the end, and K with an odd number of 64-wide blocks.  Against the oracle, and the bits of the tile
    the library would take."""
    if tile[1] == 32 and epi < 2:
        with pytest.raises(xb.XemaError) as e:
            _gemm_case(np.random.default_rng(1), 1, 40, 512, 192, epi, tile=tile)
        assert e.value.status == xb.XEMA_EINVAL
        return
    for rows in (1, 31, 33, 96, 127, 128, 129, 160, 225, 257):
        got, ref = _gemm_case(np.random.default_rng(300 + rows + epi), 2, rows, 512, 192, epi, tile=tile)
        if epi == xb.EPI_GATE_RES_F32:
            assert_close(got, ref, ("gemm edges", epi, rows, tile), rel=1e-4, cos=0.9999999)
        else:
            assert_bf16_close(got, ref, ("gemm edges", epi, rows, tile), atol_rms=2e-3 if epi == xb.EPI_BIAS_GELU else 2e-4)
        assert np.array_equal(got, _gemm_case(np.random.default_rng(300 + rows + epi), 2, rows, 512, 192, epi)[0]), (rows, tile)


@pytest.mark.parametrize("N,K", [(512, 320), (1536, 64), (768, 448), (1536, 1600)])
def test_gemm_tile_forms_give_the_same_bits(N, K):
    """The tile is chosen from the size of the problem; a row's bits must not show it.  A problem that
    gives every CTA several tiles, in every tile form and in the one the library takes, and part of
    its rows as problems of their own; K with an odd number of 64-wide blocks (a stage of the smaller
    forms holds two); a small one also against the oracle."""
    rng = np.random.default_rng(12 + N)
    rows = 256 * (2 * 74 * 256 // N + 1)
    a_dev, w_dev, b_dev = (to_dev(rand_bf16(rng, s, c)[0]) for s, c in (((rows, K), 1.0), ((N, K), 0.05), ((N,), 0.5)))
    gate = torch.from_numpy(rng.standard_normal(N, dtype=np.float32)).to(DEV)
    res = torch.from_numpy(rng.standard_normal((rows, N), dtype=np.float32)).to(DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)

    def run(n, epi, tile=None):
        out = torch.zeros(n, N, dtype=torch.int16, device=DEV)
        kw = dict(status=status.data_ptr(), a=a_dev.data_ptr(), lda=K, a_batch_rows=n, w=w_dev.data_ptr(), ldw=K,
                  bias=b_dev.data_ptr(), out=out.data_ptr(), ldo=N, out_batch_rows=n, batch=1, rows=n, N=N, K=K,
                  epilogue=epi, resid=res.data_ptr(), ldr=N, resid_batch_rows=n, gate=gate.data_ptr(), gate_stride=N)
        if tile is None:
            xb.xema_op_gemm(**kw)
        else:
            xb.xema_op_gemm_in_tile(*tile, **kw)
        return out

    for epi in (xb.EPI_BIAS, xb.EPI_GATE_RES_BF16):
        full = run(rows, epi)
        for tile in TILES:
            if N % tile[1] == 0 and (tile[1] > 32 or epi == xb.EPI_GATE_RES_BF16):
                assert torch.equal(run(rows, epi, tile), full), (epi, tile)
        for n in (100, 1300, 3000):
            if n < rows:
                assert torch.equal(run(n, epi), full[:n]), (epi, n)
    _sync_status(status)
    got, ref = _gemm_case(rng, 1, 100, N, K, xb.EPI_BIAS)
    assert_bf16_close(got, ref, ("gemm small tile", N, K), atol_rms=2e-4)


@pytest.mark.parametrize("epi", [xb.EPI_GATE_RES_F32, xb.EPI_GATE_RES_BF16])
@pytest.mark.parametrize("rows,N", [(1, 256), (37, 384), (300, 512), (700, 1536)])
def test_gemm_residual_rows_may_be_shared(epi, rows, N):
    """ldr = 0: one residual row for all; resid_batch_rows = 0: the same rows for every batch element;
    overlapping residual rows; one row with no row stride at all.  The same bits as with the residual
    written out."""
    rng = np.random.default_rng(60 + rows)
    B, K = 2, 128
    a_dev, w_dev, b_dev = (to_dev(rand_bf16(rng, s, c)[0]) for s, c in (((B, rows, K), 1.0), ((N, K), 0.05), ((N,), 0.5)))
    gate = torch.from_numpy(rng.standard_normal((B, N), dtype=np.float32)).to(DEV)
    f32 = epi == xb.EPI_GATE_RES_F32
    flat = torch.from_numpy(rng.standard_normal(B * rows * N + N, dtype=np.float32)).to(DEV)
    flat = flat.to(torch.bfloat16) if f32 else flat
    status = torch.zeros(1, dtype=torch.int32, device=DEV)

    def run(resid, ldr, batch_rows, batch=B, ldo=N):
        out = torch.zeros(B, rows, N, dtype=torch.float32 if f32 else torch.bfloat16, device=DEV)
        xb.xema_op_gemm(status=status.data_ptr(), a=a_dev.data_ptr(), lda=K, a_batch_rows=rows, w=w_dev.data_ptr(), ldw=K,
                        bias=b_dev.data_ptr(), out=out.data_ptr(), ldo=ldo, out_batch_rows=rows if batch > 1 else 0, batch=batch,
                        rows=rows, N=N, K=K, epilogue=epi, resid=resid.data_ptr(), ldr=ldr, resid_batch_rows=batch_rows,
                        gate=gate.data_ptr(), gate_stride=N)
        return out

    one_row = flat[:N].expand(B, rows, N).contiguous()
    same_rows = flat[:rows * N].view(1, rows, N).expand(B, rows, N).contiguous()
    assert torch.equal(run(flat, 0, rows), run(one_row, N, rows)) and torch.equal(run(flat, 0, 0), run(one_row, N, rows))
    assert torch.equal(run(flat, N, 0), run(same_rows, N, rows))
    windows = flat.as_strided((B, rows, N), (rows * 64, 64, 1)).contiguous()
    assert torch.equal(run(flat, 64, rows), run(windows, N, rows))
    if rows == 1:
        assert torch.equal(run(flat, 0, 0, batch=1, ldo=0)[:1], run(flat, N, 1, batch=1)[:1])
    _sync_status(status)


@pytest.mark.parametrize("rows", [256 * 49 + 1, 256 * 51 - 31])
def test_gemm_wide_gated_tile_with_many_tiles_per_pair(rows):
    """More than four 256 x 256 tiles a CTA pair, where the fp32-out gated form runs with another ring of residual
    chunks: the bits of the 256 x 128 tile, K blocks fewer and more than its stages, the last rows against
    the oracle (tolerance as in test_gemm_epilogues) and rows past the end untouched."""
    N = 1536
    rng = np.random.default_rng(70 + rows)
    for K in (64, 448, 832):
        a_dev, w_dev, b_dev = (to_dev(rand_bf16(rng, s, c)[0]) for s, c in (((rows, K), 1.0), ((N, K), 0.05), ((N,), 0.5)))
        gate = torch.from_numpy(rng.standard_normal(N, dtype=np.float32)).to(DEV)
        res = to_dev(rand_bf16(rng, (rows, N))[0])
        status = torch.zeros(1, dtype=torch.int32, device=DEV)

        def run(tile):
            out = torch.full((rows + 5, N), float("nan"), device=DEV)
            xb.xema_op_gemm_in_tile(*tile, status=status.data_ptr(), a=a_dev.data_ptr(), lda=K, a_batch_rows=rows,
                                    w=w_dev.data_ptr(), ldw=K, bias=b_dev.data_ptr(), out=out.data_ptr(), ldo=N,
                                    out_batch_rows=rows, batch=1, rows=rows, N=N, K=K, epilogue=xb.EPI_GATE_RES_F32,
                                    resid=res.data_ptr(), ldr=N, resid_batch_rows=rows, gate=gate.data_ptr(), gate_stride=N)
            return out

        wide, narrow = run((1, 256)), run((1, 128))
        _sync_status(status)
        assert torch.equal(wide[:rows], narrow[:rows]) and bool(wide[rows:].isnan().all())
        c = slice(rows - 300, rows)
        as64 = lambda t: t.view(torch.bfloat16).double()
        ref = as64(res[c]) + gate.double() * (as64(a_dev[c]) @ as64(w_dev).T + as64(b_dev))
        assert_close(wide[c].cpu().numpy(), ref.cpu().numpy(), ("gemm many wide tiles", rows, K), rel=1e-4, cos=0.9999999)


def test_gemm_many_tiles_persistent():
    """More tiles than SMs so every CTA runs several tiles through both TMEM accumulators."""
    rng = np.random.default_rng(7)
    got, ref = _gemm_case(rng, 1, 2222, 6144, 512, xb.EPI_BIAS)
    assert_bf16_close(got, ref, "gemm persistent", atol_rms=2e-4)


def test_gemm_rows_are_chunk_invariant():
    """The same rows computed as part of a large and of a small, offset problem: identical bits."""
    rng = np.random.default_rng(8)
    rows, N, K = 700, 512, 1024
    ab, _ = rand_bf16(rng, (1, rows, K))
    wb, _ = rand_bf16(rng, (N, K), 0.05)
    bb, _ = rand_bf16(rng, (N,), 0.5)
    a_dev, w_dev, b_dev = to_dev(ab), to_dev(wb), to_dev(bb)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    full = torch.zeros(1, rows, N, dtype=torch.int16, device=DEV)
    common = dict(lda=K, w=w_dev.data_ptr(), ldw=K, bias=b_dev.data_ptr(), ldo=N, batch=1, N=N, K=K,
                  epilogue=xb.EPI_BIAS_GELU)
    xb.xema_op_gemm(status=status.data_ptr(), a=a_dev.data_ptr(), a_batch_rows=rows, out=full.data_ptr(),
                    out_batch_rows=rows, rows=rows, **common)
    r0, n = 233, 301
    part = torch.zeros(1, n, N, dtype=torch.int16, device=DEV)
    xb.xema_op_gemm(status=status.data_ptr(), a=a_dev.data_ptr() + r0 * K * 2, a_batch_rows=n, out=part.data_ptr(),
                    out_batch_rows=n, rows=n, **common)
    _sync_status(status)
    assert torch.equal(full[:, r0:r0 + n], part)


def _exponent_units(q_f32, dh):
    """What the Q projection's fused epilogue hands the attention: q multiplied by
    log2(e) / sqrt(dh) in float32 and rounded to bf16 once.  Returns (bits, the exact float64 q
    those bits stand for)."""
    c = np.float32(xb.exponent_scale(dh))
    bits = bf16_bits(q_f32.astype(np.float32) * c)
    return bits, bits_to_f64(bits) / np.float64(c)


def _attention_case(rng, B, rows, keys, H, dh, q_scale=1.0):
    D = H * dh
    qb, qf = _exponent_units(rng.standard_normal((B, rows, D), dtype=np.float32) * np.float32(q_scale), dh)
    kvb, kvf = rand_bf16(rng, (B, keys, 2 * D))
    q_dev, kv_dev = to_dev(qb), to_dev(kvb)
    o = torch.full((B, rows, D), 0x7FC0, dtype=torch.int16, device=DEV)
    lse = torch.full((B, H, rows), float("nan"), dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    xb.xema_op_attention(q_dev.data_ptr(), D, rows, kv_dev.data_ptr(), kv_dev.data_ptr() + D * 2, 2 * D, keys,
                         o.data_ptr(), lse.data_ptr(), B, rows, keys, H, dh, status=status.data_ptr(), q_scale=1.0)
    _sync_status(status)
    ref_o = np.empty((B, rows, H, dh))
    ref_l = np.empty((B, H, rows))
    for b in range(B):
        for h in range(H):
            ref_o[b, :, h], ref_l[b, h] = ob.attention_head(qf[b, :, h * dh:(h + 1) * dh],
                                                            kvf[b, :, h * dh:(h + 1) * dh],
                                                            kvf[b, :, D + h * dh:D + (h + 1) * dh], 1 / math.sqrt(dh))
    return from_dev_bf16(o), ref_o.reshape(B, rows, D), lse.cpu().numpy(), ref_l


@pytest.mark.parametrize("B,rows,keys,H,dh", [(1, 128, 128, 1, 64), (1, 128, 256, 2, 64), (1, 200, 500, 3, 64),
                                              (2, 77, 1000, 2, 64), (1, 144, 288, 8, 64), (1, 300, 2222, 2, 64),
                                              (1, 128, 128, 1, 128), (2, 150, 700, 2, 128)])
def test_attention(B, rows, keys, H, dh):
    rng = np.random.default_rng(200 + rows + keys)
    got_o, ref_o, got_l, ref_l = _attention_case(rng, B, rows, keys, H, dh)
    assert_bf16_close(got_o, ref_o, ("attention o", B, rows, keys, H, dh), atol_rms=1.5e-2, cos=0.9999)
    assert np.abs(got_l - ref_l).max() < 2e-3


@pytest.mark.parametrize("dh", [64, 128])
@pytest.mark.parametrize("rows,keys", [(1, 1), (127, 64), (128, 65), (129, 127), (256, 129), (257, 511), (33, 512), (300, 513)])
def test_attention_edges(rows, keys, dh):
    """Rows and keys at the edges of 32-row warps, 128-row tiles, two-tile items, 64-key halves and
    128-key blocks, on both sides of the block count from which whole blocks run without masking.
    Tolerances as in test_attention."""
    rng = np.random.default_rng(700 + rows + keys)
    got_o, ref_o, got_l, ref_l = _attention_case(rng, 2, rows, keys, 3, dh)
    assert_bf16_close(got_o, ref_o, ("attention edges", rows, keys, dh), atol_rms=1.5e-2, cos=0.9999)
    assert np.abs(got_l - ref_l).max() < 2e-3


@pytest.mark.parametrize("dh,keys,spread,o_max,lse_max", [(64, 4608, 1.0, 2.4e-3, 1.5e-6), (128, 40, 1.0, 2.2e-3, 5e-7),
                                                          (128, 288, 1.0, 2.3e-3, 5e-7), (128, 600, 3.0, 2.1e-3, 2e-6)])
def test_attention_rms_error(dh, keys, spread, o_max, lse_max):
    """Root-mean-square error of o (relative) and of lse over a million elements, where an element-wise bound
    sees little.  Rounding o to bf16 alone gives 1.66e-3 and rounding independent probabilities to bf16 as
    much again, 2.35e-3 together.  head_dim 128 has to stay below that where a few keys carry a row (few
    keys, or scores spread threefold), because its largest probabilities are exact or cancel: half-way between
    2.35e-3 and the 2.05e-3, 2.24e-3 and 1.92e-3 it reaches.  lse is a sum of fp32 exponentials: its bound is two to
    three times what ex2 of 2^-22 gives (the error of a score of size s adds s * 2^-24), and for head_dim 64 less
    than the 2.2e-6 that exponentials with a common error of 5e-6 in 14 of 32 places would add up to."""
    gen = torch.Generator(device=DEV).manual_seed(5)
    rows, H = (500, 16) if keys > 1000 else (288, 96)
    D = H * dh
    q = (torch.randn(rows, D, device=DEV, generator=gen) * (spread * xb.exponent_scale(dh))).to(torch.bfloat16)
    kv = torch.randn(keys, 2 * D, device=DEV, generator=gen).to(torch.bfloat16)
    o = torch.empty(rows, D, dtype=torch.bfloat16, device=DEV)
    lse = torch.empty(H, rows, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    xb.xema_op_attention(q.data_ptr(), D, rows, kv.data_ptr(), kv.data_ptr() + D * 2, 2 * D, keys, o.data_ptr(), lse.data_ptr(),
                         1, rows, keys, H, dh, status=status.data_ptr(), q_scale=1.0)
    _sync_status(status)
    err = ref = lse_err = 0.0
    for h in range(H):
        c = slice(h * dh, (h + 1) * dh)
        s = (q[:, c].double() @ kv[:, c].double().T) * math.log(2.0)
        want = torch.softmax(s, -1) @ kv[:, D + h * dh:D + (h + 1) * dh].double()
        err += (o[:, c].double() - want).square().sum().item()
        ref += want.square().sum().item()
        lse_err += (lse[h].double() - torch.logsumexp(s, -1)).square().mean().item() / H
    assert math.sqrt(err / ref) < o_max and math.sqrt(lse_err) < lse_max, (math.sqrt(err / ref), math.sqrt(lse_err))


@pytest.mark.parametrize("dh", [64, 128])
@pytest.mark.parametrize("plain", [False, True])
def test_attention_non_finite_keys_reach_their_rows(dh, plain):
    """A key that holds a NaN makes every row of its head NaN, one that holds an infinity the rows whose score
    for it is +infinity (the others give it probability 0), whichever place of a key block it has -- all
    places between two multiples of 64 are tried, because different places take different exponentials.
    Heads without such a key are not touched."""
    rng = np.random.default_rng(15)
    rows, keys, H = 140, 300, 66
    D = H * dh
    q, kv = rng.standard_normal((rows, D)), bf16_bits(rng.standard_normal((keys, 2 * D), dtype=np.float32))
    qb, qf = (lambda b: (b, bits_to_f64(b)))(bf16_bits(q.astype(np.float32))) if plain else _exponent_units(q, dh)
    for h in range(64):
        at = 64 * (h % 4) + h
        if at < keys:
            kv[at, h * dh + 3] = 0x7FC0 if h % 2 else 0x7F80
    kvf = bits_to_f64(kv)
    q_dev, kv_dev = to_dev(qb), to_dev(kv)
    o = torch.zeros(rows, D, dtype=torch.int16, device=DEV)
    lse = torch.zeros(H, rows, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    xb.xema_op_attention(q_dev.data_ptr(), D, rows, kv_dev.data_ptr(), kv_dev.data_ptr() + D * 2, 2 * D, keys, o.data_ptr(),
                         lse.data_ptr(), 1, rows, keys, H, dh, status=status.data_ptr(), q_scale=None if plain else 1.0)
    _sync_status(status)
    got, got_l = from_dev_bf16(o), lse.cpu().numpy()
    for h in range(H):
        c = slice(h * dh, (h + 1) * dh)
        with np.errstate(invalid="ignore"):
            s = qf[:, c] @ kvf[:, c].T / math.sqrt(dh)
            bad = np.isnan(s).any(axis=1) | np.isposinf(s).any(axis=1)
        assert np.array_equal(np.isnan(got[:, c]).all(axis=1), bad) and np.array_equal(np.isnan(got[:, c]).any(axis=1), bad), h
        assert np.array_equal(np.isfinite(got_l[h]), ~bad), h
        ok = ~bad
        if ok.any():
            e = np.exp(s[ok] - s[ok].max(axis=1, keepdims=True))
            want = (e / e.sum(axis=1, keepdims=True)) @ kvf[:, D + h * dh:D + (h + 1) * dh]
            assert_bf16_close(got[ok][:, c], want, ("non-finite keys", dh, h), atol_rms=1.5e-2, cos=0.9999)


@pytest.mark.parametrize("dh", [64, 128])
def test_attention_items_of_one_cta_with_flagged_rows(dh):
    """More work items than SMs, so that CTAs run several; the scores of a few heads lie near +-260 (in
    exponents to base 2), so first and later items of some CTAs have to be repeated against their rows'
    maxima while the other items keep their results.  Tolerances as in
    test_attention_dh64_scores_far_from_zero (lse relative to its size)."""
    rng = np.random.default_rng(93 + dh)
    rows, keys, H = 130, 300, 170
    D = H * dh
    far = {3: 260.0, 20: -260.0, 151: 260.0, 168: -260.0}
    q = rng.standard_normal((1, rows, D))
    kv = rng.standard_normal((1, keys, 2 * D))
    u = np.ones(dh) / math.sqrt(dh)
    a = 30.0
    for h, offset in far.items():
        c = slice(h * dh, (h + 1) * dh)
        q[0, :, c] = a * u + 0.3 * rng.standard_normal((rows, dh))
        kv[0, :, c] = offset * math.sqrt(dh) / 1.4426950408889634 / a * u + 0.3 * rng.standard_normal((keys, dh))
    (qb, qf), kvb = _exponent_units(q, dh), bf16_bits(kv.astype(np.float32))
    kvf = bits_to_f64(kvb)
    q_dev, kv_dev = to_dev(qb), to_dev(kvb)
    o = torch.zeros(1, rows, D, dtype=torch.int16, device=DEV)
    lse = torch.zeros(1, H, rows, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    xb.xema_op_attention(q_dev.data_ptr(), D, rows, kv_dev.data_ptr(), kv_dev.data_ptr() + D * 2, 2 * D, keys,
                         o.data_ptr(), lse.data_ptr(), 1, rows, keys, H, dh, status=status.data_ptr(), q_scale=1.0)
    _sync_status(status)
    got = from_dev_bf16(o)
    for h in sorted(set(far) | {0, 2, 4, 19, 21, 147, 148, 150, 152, 167, 169}):
        c = slice(h * dh, (h + 1) * dh)
        ref_o, ref_l = ob.attention_head(qf[0, :, c], kvf[0, :, c], kvf[0, :, D + h * dh:D + (h + 1) * dh], 1 / math.sqrt(dh))
        assert_bf16_close(got[0, :, c], ref_o, ("flagged items", dh, h), atol_rms=2.5e-2, cos=0.9998)
        assert np.abs(lse.cpu().numpy()[0, h] - ref_l).max() < 2e-3 * max(1.0, np.abs(ref_l).max() / 10)


@pytest.mark.parametrize("dh", [64, 128])
def test_attention_rows_do_not_depend_on_tiles_per_item(dh):
    """500 rows of 60 heads run as items of two tiles, 211 of them as items of one: the same bits."""
    rng = np.random.default_rng(94)
    rows, keys, H = 500, 700, 60
    D = H * dh
    q_dev, kv_dev = to_dev(_exponent_units(rng.standard_normal((1, rows, D)), dh)[0]), to_dev(rand_bf16(rng, (1, keys, 2 * D))[0])
    status = torch.zeros(1, dtype=torch.int32, device=DEV)

    def run(r0, n):
        o = torch.zeros(n, D, dtype=torch.int16, device=DEV)
        lse = torch.zeros(H, n, dtype=torch.float32, device=DEV)
        xb.xema_op_attention(q_dev.data_ptr() + r0 * D * 2, D, n, kv_dev.data_ptr(), kv_dev.data_ptr() + D * 2, 2 * D, keys,
                             o.data_ptr(), lse.data_ptr(), 1, n, keys, H, dh, status=status.data_ptr(), q_scale=1.0)
        return o, lse

    (o_all, l_all), (o_part, l_part) = run(0, rows), run(167, 211)
    _sync_status(status)
    assert torch.equal(o_all[167:167 + 211], o_part) and torch.equal(l_all[:, 167:167 + 211], l_part)


def test_attention_peaked_scores():
    """Large |q| makes the softmax peaked and takes many scores out of the polynomial's range."""
    rng = np.random.default_rng(9)
    got_o, ref_o, got_l, ref_l = _attention_case(rng, 1, 256, 1500, 2, 64, q_scale=6.0)
    assert_bf16_close(got_o, ref_o, "attention peaked", atol_rms=1.5e-2, cos=0.9999)
    assert np.abs(got_l - ref_l).max() < 5e-3 * max(1.0, np.abs(ref_l).max())


@pytest.mark.parametrize("dh", [64, 128])
def test_attention_with_a_plain_q(dh):
    """A q that was not multiplied beforehand: the library is told the scale and multiplies the fp32
    scores by it, so nothing is rounded that a prepared q would not have rounded.  Tolerances as in
    test_attention."""
    rng = np.random.default_rng(44 + dh)
    B, rows, keys, H = 1, 200, 700, 2
    D = H * dh
    qb, qf = rand_bf16(rng, (B, rows, D))
    kvb, kvf = rand_bf16(rng, (B, keys, 2 * D))
    q_dev, kv_dev = to_dev(qb), to_dev(kvb)
    o = torch.full((B, rows, D), 0x7FC0, dtype=torch.int16, device=DEV)
    lse = torch.full((B, H, rows), float("nan"), dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    xb.xema_op_attention(q_dev.data_ptr(), D, rows, kv_dev.data_ptr(), kv_dev.data_ptr() + D * 2, 2 * D, keys,
                         o.data_ptr(), lse.data_ptr(), B, rows, keys, H, dh, status=status.data_ptr())
    _sync_status(status)
    got = from_dev_bf16(o)
    for h in range(H):
        ref_o, ref_l = ob.attention_head(qf[0, :, h * dh:(h + 1) * dh], kvf[0, :, h * dh:(h + 1) * dh],
                                         kvf[0, :, D + h * dh:D + (h + 1) * dh], 1 / math.sqrt(dh))
        assert_bf16_close(got[0, :, h * dh:(h + 1) * dh], ref_o, ("plain q", dh, h), atol_rms=1.5e-2, cos=0.9999)
        assert np.abs(lse.cpu().numpy()[0, h] - ref_l).max() < 2e-3


def test_attention_rows_are_chunk_invariant():
    rng = np.random.default_rng(10)
    B, rows, keys, H, dh = 1, 500, 900, 2, 64
    D = H * dh
    qb, _ = rand_bf16(rng, (B, rows, D), 2.0)
    kvb, _ = rand_bf16(rng, (B, keys, 2 * D))
    q_dev, kv_dev = to_dev(qb), to_dev(kvb)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)

    def run(r0, n):
        o = torch.zeros(B, n, D, dtype=torch.int16, device=DEV)
        lse = torch.zeros(B, H, n, dtype=torch.float32, device=DEV)
        xb.xema_op_attention(q_dev.data_ptr() + r0 * D * 2, D, n, kv_dev.data_ptr(), kv_dev.data_ptr() + D * 2, 2 * D,
                             keys, o.data_ptr(), lse.data_ptr(), B, n, keys, H, dh, status=status.data_ptr())
        return o, lse

    o_all, l_all = run(0, rows)
    o_part, l_part = run(167, 211)
    _sync_status(status)
    assert torch.equal(o_all[:, 167:167 + 211], o_part)
    assert torch.equal(l_all[:, :, 167:167 + 211], l_part)


@pytest.mark.parametrize("name,norm_all", [("tiny", True), ("tiny", False), ("flux", True), ("flux", False)])
def test_gemm_epilogue_rmsnorm_rope(name, norm_all):
    """Linear + per-head RMSNorm * gain + RoPE fused in the GEMM epilogue: the Q product
    (every head) and the K|V product (heads of the first half only)."""
    t = template(name)
    dh = t.head_dim
    rng = np.random.default_rng(31 + dh + norm_all)
    H, K, rows, pos0, B = 4, 192, 200, t.s_text - 20, 2         # rows span the text / video boundary
    Dh = H * dh
    N = Dh if norm_all else 2 * Dh
    ab, af = rand_bf16(rng, (B, rows, K))
    wb, wf = rand_bf16(rng, (N, K), 0.08)
    bb, bf = rand_bf16(rng, (N,), 0.3)
    gb, gf = rand_bf16(rng, (dh,), 1.0)
    a_dev, w_dev, b_dev, g_dev = to_dev(ab), to_dev(wb), to_dev(bb), to_dev(gb)
    rope = torch.from_numpy(xb.xema_rope_table(xb.make_config(t))).to(DEV)
    out = torch.full((B, rows, N), 0x7FC0, dtype=torch.int16, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    xb.xema_op_gemm(status=status.data_ptr(), a=a_dev.data_ptr(), lda=K, a_batch_rows=rows, w=w_dev.data_ptr(), ldw=K,
                    bias=b_dev.data_ptr(), out=out.data_ptr(), ldo=N, out_batch_rows=rows, batch=B, rows=rows, N=N,
                    K=K, epilogue=xb.EPI_BIAS_NORM_ROPE, head_dim=dh, norm_cols=Dh, rope_pos0=pos0, rms_eps=1e-6,
                    norm_gain=g_dev.data_ptr(), rope=rope.data_ptr())
    _sync_status(status)
    acc = af @ wf.T + bf
    ang = ob.rope_angles(t)[pos0:pos0 + rows]
    ref = acc.copy()
    for b in range(B):
        v = acc[b, :, :Dh].reshape(rows, H, dh)
        ref[b, :, :Dh] = ob.apply_rope(ob.rms_norm(v, gf, 1e-6), ang).reshape(rows, Dh)
    assert_bf16_close(from_dev_bf16(out), ref, ("gemm norm+rope", name, norm_all), atol_rms=3e-4)


@pytest.mark.parametrize("name", ["tiny", "flux"])
@pytest.mark.parametrize("tile", TILES[:4])
def test_gemm_epilogue_rmsnorm_rope_in_every_tile(name, tile):
    """The same epilogue with the tile named, rows at the edges of warps and tiles, two batch elements, a
    K|V product whose norm ends inside a 256-column tile or between two: against the oracle, and the
    bits of the tile the library would take."""
    t = template(name)
    dh = t.head_dim
    K, N, B, pos0 = 192, 768, 2, t.s_text - 20
    rng = np.random.default_rng(33 + dh)
    wb, wf = rand_bf16(rng, (N, K), 0.08)
    bb, bf = rand_bf16(rng, (N,), 0.3)
    gb, gf = rand_bf16(rng, (dh,), 1.0)
    rope = torch.from_numpy(xb.xema_rope_table(xb.make_config(t))).to(DEV)
    w_dev, b_dev, g_dev = to_dev(wb), to_dev(bb), to_dev(gb)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    for rows, norm in ((1, 512), (33, 384), (128, 512), (160, 768), (257, 384)):
        ab, af = rand_bf16(rng, (B, rows, K))
        a_dev = to_dev(ab)

        def run(in_tile):
            out = torch.full((B, rows + 3, N), 0x7FC0, dtype=torch.int16, device=DEV)
            kw = dict(status=status.data_ptr(), a=a_dev.data_ptr(), lda=K, a_batch_rows=rows, w=w_dev.data_ptr(), ldw=K,
                      bias=b_dev.data_ptr(), out=out.data_ptr(), ldo=N, out_batch_rows=rows + 3, batch=B, rows=rows, N=N, K=K,
                      epilogue=xb.EPI_BIAS_NORM_ROPE, head_dim=dh, norm_cols=norm, rope_pos0=pos0, rms_eps=1e-6,
                      norm_gain=g_dev.data_ptr(), rope=rope.data_ptr())
            if in_tile is None:
                xb.xema_op_gemm(**kw)
            else:
                xb.xema_op_gemm_in_tile(*in_tile, **kw)
            return out

        if tile[1] < dh:
            with pytest.raises(xb.XemaError) as e:
                run(tile)
            assert e.value.status == xb.XEMA_EINVAL
            return
        out = run(tile)
        assert torch.equal(out, run(None)), (rows, norm)
        _sync_status(status)
        assert (out[:, rows:] == 0x7FC0).all()
        ref = af @ wf.T + bf
        for b in range(B):
            v = ref[b, :, :norm].reshape(rows, norm // dh, dh)
            ref[b, :, :norm] = ob.apply_rope(ob.rms_norm(v, gf, 1e-6), ob.rope_angles(t)[pos0:pos0 + rows]).reshape(rows, norm)
        assert_bf16_close(from_dev_bf16(out[:, :rows]), ref, ("gemm norm+rope", name, tile, rows, norm), atol_rms=3e-4)


@pytest.mark.parametrize("offset", [-260.0, -100.0, 100.0, 260.0])
def test_attention_dh64_scores_far_from_zero(offset):
    """Every score of a row lies near `offset` (in exponents to base 2), with a spread of a few
    units: far below zero the unnormalised probabilities underflow, far above they overflow, and
    in between (|offset| = 100) the sums leave the range the kernel trusts.  The head_dim-64
    kernel forms 2^score without a reference in its first pass, so all of these must be caught
    by its range check and repeated against the row's true maximum; rows of an ordinary head in
    the same launch are unaffected."""
    rng = np.random.default_rng(91)
    B, rows, keys, H, dh = 1, 300, 700, 2, 64
    D = H * dh
    u = rng.standard_normal(dh)
    u /= np.linalg.norm(u)
    q = rng.standard_normal((B, rows, D))
    kv = rng.standard_normal((B, keys, 2 * D))
    # head 0: q = a u + noise, k = b u + noise with a * b / 8 * log2(e) = offset
    a = 30.0
    b = offset * 8.0 / 1.4426950408889634 / a
    q[0, :, :dh] = a * u + 0.3 * rng.standard_normal((rows, dh))
    kv[0, :, :dh] = b * u + 0.3 * rng.standard_normal((keys, dh))
    (qb, qf), kvb = _exponent_units(q, dh), bf16_bits(kv.astype(np.float32))
    kvf = bits_to_f64(kvb)
    q_dev, kv_dev = to_dev(qb), to_dev(kvb)
    o = torch.zeros(B, rows, D, dtype=torch.int16, device=DEV)
    lse = torch.zeros(B, H, rows, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    xb.xema_op_attention(q_dev.data_ptr(), D, rows, kv_dev.data_ptr(), kv_dev.data_ptr() + D * 2, 2 * D, keys,
                         o.data_ptr(), lse.data_ptr(), B, rows, keys, H, dh, status=status.data_ptr(), q_scale=1.0)
    _sync_status(status)
    got = from_dev_bf16(o)
    expo = (qf[0, :, :dh] @ kvf[0, :, :dh].T) / math.sqrt(dh) * 1.4426950408889634
    assert abs(np.median(expo) - offset) < 0.1 * abs(offset) and expo.max() - expo.min() > 10
    for h in range(H):
        ref_o, ref_l = ob.attention_head(qf[0, :, h * dh:(h + 1) * dh], kvf[0, :, h * dh:(h + 1) * dh],
                                         kvf[0, :, D + h * dh:D + (h + 1) * dh], 1 / math.sqrt(dh))
        assert_bf16_close(got[0, :, h * dh:(h + 1) * dh], ref_o, ("scores far from zero", offset, h), atol_rms=2e-2, cos=0.9999)
        assert np.abs(lse.cpu().numpy()[0, h] - ref_l).max() < 1e-3 * max(np.abs(ref_l).max(), 1.0)


def test_attention_dh64_rows_keep_their_bits_when_neighbours_repeat():
    """Rows 128..255 get scores in the hundreds and have their item (a tile here, as there are SMs enough)
    repeated; the rows of the other items must come out with exactly the bits they have when nothing
    repeats.  (Quiet rows inside a repeated item: the next test.)"""
    rng = np.random.default_rng(17)
    B, rows, keys, H, dh = 1, 384, 900, 1, 64
    q = rng.standard_normal((B, rows, dh))
    kv = rng.standard_normal((B, keys, 2 * dh))
    loud = q.copy()
    loud[0, 128:256] *= 60.0                                   # exponents of +-300 and more
    kvb = bf16_bits(kv.astype(np.float32))
    kv_dev = to_dev(kvb)
    outs = []
    for qq in (q, loud):
        qb, _ = _exponent_units(qq, dh)
        q_dev = to_dev(qb)
        o = torch.zeros(B, rows, dh, dtype=torch.int16, device=DEV)
        lse = torch.zeros(B, H, rows, dtype=torch.float32, device=DEV)
        status = torch.zeros(1, dtype=torch.int32, device=DEV)
        xb.xema_op_attention(q_dev.data_ptr(), dh, rows, kv_dev.data_ptr(), kv_dev.data_ptr() + dh * 2, 2 * dh, keys,
                             o.data_ptr(), lse.data_ptr(), B, rows, keys, H, dh, status=status.data_ptr(), q_scale=1.0)
        _sync_status(status)
        outs.append((o.cpu().numpy(), lse.cpu().numpy()))
    (o0, l0), (o1, l1) = outs
    quiet = np.r_[0:128, 256:rows]
    assert np.array_equal(o0[:, quiet], o1[:, quiet]) and np.array_equal(l0[:, :, quiet], l1[:, :, quiet])
    assert not np.array_equal(o0[:, 128:256], o1[:, 128:256])
    assert np.isfinite(l1).all()


@pytest.mark.parametrize("dh", [64, 128])
def test_attention_quiet_rows_of_a_repeated_item_keep_their_bits(dh):
    """384 rows of 60 heads: more tiles than SMs, so items of two tiles, the last of each head with one
    wholly past the end.  In some heads single rows, in others a whole tile get scores far out of the
    trusted range (for head_dim 128: far above the first block's largest), so their items are repeated; every
    other row of those items must come out with exactly the bits it has when nothing repeats, and the
    loud rows right (tolerances as in test_attention_scores_growing_along_the_keys)."""
    rng = np.random.default_rng(18 + dh)
    rows, keys, H = 384, 700, 60
    D = H * dh
    q = rng.standard_normal((rows, D))
    kv = bf16_bits(rng.standard_normal((keys, 2 * D), dtype=np.float32))
    kvf = bits_to_f64(kv)
    loud = {1: [5], 7: [70, 127], 20: [128, 200], 33: list(range(128, 256)), 40: list(range(0, 128)), 58: [0, 383], 59: [300]}
    q_loud = q.copy()
    for h, rs in loud.items():
        q_loud[rs, h * dh:(h + 1) * dh] *= 60.0 if dh == 64 else 400.0
    kv_dev = to_dev(kv)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    outs = []
    for qq in (q, q_loud):
        qb, qf = _exponent_units(qq, dh)
        q_dev = to_dev(qb)
        o = torch.zeros(rows, D, dtype=torch.int16, device=DEV)
        lse = torch.zeros(H, rows, dtype=torch.float32, device=DEV)
        xb.xema_op_attention(q_dev.data_ptr(), D, rows, kv_dev.data_ptr(), kv_dev.data_ptr() + D * 2, 2 * D, keys, o.data_ptr(),
                             lse.data_ptr(), 1, rows, keys, H, dh, status=status.data_ptr(), q_scale=1.0)
        _sync_status(status)
        outs.append((o.view(rows, H, dh), lse))
    (o0, l0), (o1, l1) = outs
    quiet = torch.ones(rows, H, dtype=torch.bool, device=DEV)
    for h, rs in loud.items():
        quiet[rs, h] = False
    assert torch.equal(o0[quiet], o1[quiet]) and torch.equal(l0.T[quiet], l1.T[quiet])
    got, got_l = from_dev_bf16(o1), l1.cpu().numpy()
    for h, rs in loud.items():
        c = slice(h * dh, (h + 1) * dh)
        ref_o, ref_l = ob.attention_head(qf[rs, c], kvf[:, c], kvf[:, D + h * dh:D + (h + 1) * dh], 1 / math.sqrt(dh))
        assert_bf16_close(got[rs, h], ref_o, ("loud rows", dh, h), atol_rms=2e-2, cos=0.9999)
        assert np.abs(got_l[h, rs] - ref_l).max() < 1e-3 * np.abs(ref_l).max()


@pytest.mark.parametrize("dh", [64, 128])
@pytest.mark.parametrize("rows,keys", [(1, 1), (129, 127), (256, 129), (257, 511), (300, 513)])
def test_attention_edges_in_items_of_two_tiles(rows, keys, dh):
    """The edges of test_attention_edges with heads enough (160 in two batch elements) for every item to have
    two tiles, odd tile counts included; some heads against the oracle.  Tolerances as there."""
    rng = np.random.default_rng(710 + rows + keys)
    B, H = 2, 80
    D = H * dh
    qb, qf = _exponent_units(rng.standard_normal((B, rows, D), dtype=np.float32), dh)
    kvb, kvf = rand_bf16(rng, (B, keys, 2 * D))
    q_dev, kv_dev = to_dev(qb), to_dev(kvb)
    o = torch.full((B, rows, D), 0x7FC0, dtype=torch.int16, device=DEV)
    lse = torch.full((B, H, rows), float("nan"), dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    xb.xema_op_attention(q_dev.data_ptr(), D, rows, kv_dev.data_ptr(), kv_dev.data_ptr() + D * 2, 2 * D, keys, o.data_ptr(),
                         lse.data_ptr(), B, rows, keys, H, dh, status=status.data_ptr(), q_scale=1.0)
    _sync_status(status)
    got, got_l = from_dev_bf16(o), lse.cpu().numpy()
    assert np.isfinite(got).all() and np.isfinite(got_l).all()
    for b, h in ((0, 0), (0, 41), (0, 79), (1, 0), (1, 38), (1, 79)):
        c = slice(h * dh, (h + 1) * dh)
        ref_o, ref_l = ob.attention_head(qf[b][:, c], kvf[b][:, c], kvf[b][:, D + h * dh:D + (h + 1) * dh], 1 / math.sqrt(dh))
        assert_bf16_close(got[b][:, c], ref_o, ("attention edges", rows, keys, dh, b, h), atol_rms=1.5e-2, cos=0.9999)
        assert np.abs(got_l[b, h] - ref_l).max() < 2e-3


@pytest.mark.parametrize("dh", [64, 128])
def test_attention_scores_growing_along_the_keys(dh):
    """Keys whose scores rise steadily with the key index: each block's scores lie far above the ones
    before, so every row leaves the trusted range and is repeated; and scores so far below the
    maximum that the exponentials underflow (the polynomial's clamp)."""
    rng = np.random.default_rng(77)
    B, rows, keys, H = 1, 200, 1100, 2
    D = H * dh
    u = rng.standard_normal((H, dh))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    ramp = np.linspace(-1.0, 1.0, keys)[:, None]
    q = np.empty((B, rows, D)); kv = rng.standard_normal((B, keys, 2 * D))
    for h in range(H):
        q[0, :, h * dh:(h + 1) * dh] = u[h] * 40.0 + 0.3 * rng.standard_normal((rows, dh))
        kv[0, :, h * dh:(h + 1) * dh] = u[h] * ramp * 60.0 + 0.3 * rng.standard_normal((keys, dh))
    (qb, qf), kvb = _exponent_units(q, dh), bf16_bits(kv.astype(np.float32))
    kvf = bits_to_f64(kvb)
    q_dev, kv_dev = to_dev(qb), to_dev(kvb)
    o = torch.zeros(B, rows, D, dtype=torch.int16, device=DEV)
    lse = torch.zeros(B, H, rows, dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    xb.xema_op_attention(q_dev.data_ptr(), D, rows, kv_dev.data_ptr(), kv_dev.data_ptr() + D * 2, 2 * D, keys,
                         o.data_ptr(), lse.data_ptr(), B, rows, keys, H, dh, status=status.data_ptr(), q_scale=1.0)
    _sync_status(status)
    got = from_dev_bf16(o)
    for h in range(H):
        ref_o, ref_l = ob.attention_head(qf[0, :, h * dh:(h + 1) * dh], kvf[0, :, h * dh:(h + 1) * dh],
                                         kvf[0, :, D + h * dh:D + (h + 1) * dh], 1 / math.sqrt(dh))
        # the scores span several hundred in the exp2 domain
        span = (qf[0, :, h * dh:(h + 1) * dh] @ kvf[0, :, h * dh:(h + 1) * dh].T) / math.sqrt(dh) * 1.4427
        assert span.max() - span.min() > 300
        assert_bf16_close(got[0, :, h * dh:(h + 1) * dh], ref_o, ("growing scores", dh, h), atol_rms=2e-2, cos=0.9999)
        assert np.abs(lse.cpu().numpy()[0, h] - ref_l).max() < 1e-3 * np.abs(ref_l).max()
