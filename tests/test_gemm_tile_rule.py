"""The tile that a GEMM gets (host only; without a device the rule counts a B200's 148 SMs)."""
import pytest
import torch

from paper_2607_11136_b200 import binding as xb

if torch.cuda.is_available():
    pytestmark = pytest.mark.skipif(torch.cuda.get_device_properties(0).multi_processor_count != 148, reason="148 SMs")


@pytest.mark.parametrize("batch,rows,N,K,epi,tile", [
    (1, 17776, 6144, 3072, xb.EPI_BIAS, (1, 256)), (1, 8888, 12288, 3072, xb.EPI_BIAS_GELU, (1, 256)),
    (1, 4444, 3072, 3072, xb.EPI_GATE_RES_F32, (1, 256)), (1, 2222, 3072, 3072, xb.EPI_BIAS, (1, 128)),
    (1, 1101, 1536, 6144, xb.EPI_GATE_RES_BF16, (1, 128)), (1, 333, 1024, 4096, xb.EPI_BIAS, (0, 64)),
    (1, 333, 1024, 4096, xb.EPI_GATE_RES_BF16, (0, 32)), (1, 288, 512, 2048, xb.EPI_GATE_RES_BF16, (0, 32)),
    (2, 257, 384, 192, xb.EPI_BIAS, (0, 64)), (2, 257, 512, 192, xb.EPI_GATE_RES_F32, (0, 32))])
def test_tile_rule(batch, rows, N, K, epi, tile):
    """The sizes that the rule's figures were measured at get the tile that was fastest there."""
    assert xb.xema_gemm_tile(batch=batch, rows=rows, N=N, K=K, epilogue=epi) == tile


def test_tile_rule_keeps_heads_whole_and_refuses_bad_sizes():
    for dh in (64, 128):
        for rows in (1, 300, 1101, 5000):
            assert xb.xema_gemm_tile(batch=1, rows=rows, N=512, K=512, epilogue=xb.EPI_BIAS_NORM_ROPE, head_dim=dh, norm_cols=512)[1] >= dh
    for bad in (dict(N=64), dict(K=32), dict(batch=0), dict(rows=-1), dict(epilogue=9), dict(epilogue=4, head_dim=32)):
        with pytest.raises(xb.XemaError) as e:
            xb.xema_gemm_tile(**{**dict(batch=1, rows=10, N=256, K=64, epilogue=0, norm_cols=0), **bad})
        assert e.value.status == xb.XEMA_EINVAL
