"""The shared library loads without a GPU and exports every symbol the header declares."""
import ctypes
import os
import re

from paper_2607_11136_b200 import binding as xb

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    text = open(os.path.join(ROOT, "include", "xema.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(xema_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported():
    names = _declared()
    assert len(names) >= 20
    L = ctypes.CDLL(xb.LIB_PATH)
    for n in names:
        assert hasattr(L, n), n
    assert sorted(xb.EXPORTS) == names


def test_struct_sizes_match_the_header():
    # 13 int32 + 3 float + 1 int32; name[24] + 4 x 4 + 8 + 2 x 4; 12 pointers; gemm args
    assert ctypes.sizeof(xb.xema_config) == 68
    assert ctypes.sizeof(xb.xema_tensor) == 56
    assert ctypes.sizeof(xb.xema_block_weights) == 96
    assert ctypes.sizeof(xb.xema_gemm_args) == 168


def test_gemm_layouts_that_are_refused():
    """Results whose rows or batch elements would lie over one another, and negative residual strides, are
    refused before any CUDA call; rows that nothing strides over and shared residual rows are not."""
    base = dict(a=256, lda=64, a_batch_rows=4, w=256, ldw=64, bias=256, out=256, ldo=128, out_batch_rows=4, resid=256,
                ldr=128, resid_batch_rows=4, gate=256, gate_stride=128, batch=2, rows=4, N=128, K=64, epilogue=2)
    for over, refused in ((dict(out_batch_rows=0), True), (dict(out_batch_rows=-4), True), (dict(ldo=64), True),
                          (dict(ldr=-128), True), (dict(resid_batch_rows=-1), True),
                          (dict(ldr=0), False), (dict(resid_batch_rows=0), False), (dict(ldr=0, resid_batch_rows=0), False),
                          (dict(rows=1, batch=1, ldo=0, ldr=0, out_batch_rows=0), False)):
        try:
            # (a null stream; without a driver the descriptors cannot be made, which is another status)
            args = xb.xema_gemm_args()
            for k, v in {**base, **over}.items():
                setattr(args, k, v)
            args.rows = args.rows if refused else 0     # nothing to launch
            xb._check(xb.lib().xema_op_gemm(ctypes.byref(args), None, None), "xema_op_gemm")
            status = 0
        except xb.XemaError as e:
            status = e.status
        assert (status == xb.XEMA_EINVAL) == refused, (over, status)


def test_error_paths_without_gpu():
    assert xb.version().startswith("xema-b200")
    assert xb.strerror(0) == "ok" and "budget" in xb.strerror(xb.XEMA_EBUDGET)
    from xema_inputs import template
    cfg = xb.make_config(template("tiny"))
    for bad in (0, -1, 289):
        try:
            xb.xema_trace(cfg, bad)
            raise AssertionError("expected XEMA_EINVAL")
        except xb.XemaError as e:
            assert e.status == xb.XEMA_EINVAL
    bad_cfg = xb.make_config(template("tiny"))
    bad_cfg.rope_dim_t = 15
    try:
        xb.xema_trace(bad_cfg, 1)
        raise AssertionError("expected XEMA_EINVAL")
    except xb.XemaError as e:
        assert e.status == xb.XEMA_EINVAL
    bad_cfg = xb.make_config(template("tiny"))
    bad_cfg.heads = 7
    try:
        xb.Plan(bad_cfg, 1)
        raise AssertionError("expected XEMA_EINVAL")
    except xb.XemaError as e:
        assert e.status == xb.XEMA_EINVAL
    # forward on an unbound plan is refused, not crashed
    p = xb.Plan(cfg, 2)
    assert p.launch_count() == 0
    try:
        p.block_forward(0)
        raise AssertionError("expected XEMA_ESTATE")
    except xb.XemaError as e:
        assert e.status == xb.XEMA_ESTATE
    # arena too small / misaligned / null weights are refused before any CUDA call
    w = [{k: 16 for k in xb._WEIGHT_FIELDS}]
    for arena_ptr, nbytes, want in ((256, p.peak_bytes - 1, xb.XEMA_ENOSPC), (257, p.peak_bytes, xb.XEMA_EALIGN)):
        try:
            p.bind(arena_ptr, nbytes, w, 256)
            raise AssertionError("expected an error")
        except xb.XemaError as e:
            assert e.status == want
    p.close()
