"""Which row kernel a shape takes, asked without a GPU: what a step really runs, with and without guidance."""
import ctypes as C

import pytest

from paper_2512_07503_b200 import binding as B


def _path(V, top_k, rows=(16, 64), dtype=B.SJD_BF16, flags=0, guidance=True):
    p = B.sjd_params()
    p.struct_size = C.sizeof(B.sjd_params)
    p.B, p.W, p.V, p.logits_dtype, p.top_k, p.flags = *rows, V, dtype, top_k, flags
    p.inv_temperature, p.cfg_scale = 1.0, 3.0
    p.stride_b, p.stride_w = rows[1] * V, V
    return B.sjd_row_path(p, guidance)


@pytest.mark.parametrize("guidance", [True, False])
def test_paths(guidance):
    assert _path(65536, 2000, guidance=guidance) == B.SJD_PATH_STREAM
    assert _path(65536, 8192, guidance=guidance) == B.SJD_PATH_STREAM  # a wide top-K as well
    assert _path(50264, 500, rows=(1, 8), guidance=guidance) == B.SJD_PATH_CLUSTER
    assert _path(65536, 2000, flags=B.SJD_FLAG_FORCE_GENERIC, guidance=guidance) == B.SJD_PATH_ANY_SHAPE
    assert _path(65536, 1000, flags=B.SJD_FLAG_FORCE_TILES, guidance=guidance) == B.SJD_PATH_TILES
    assert _path(1032, 7, dtype=B.SJD_F32, guidance=guidance) == B.SJD_PATH_ANY_SHAPE
    assert _path(4096, 4096, guidance=guidance) == B.SJD_PATH_ANY_SHAPE


def test_guidance_decides_how_many_blocks_share_a_row():
    # 80 rows: one array of 128 KB fits a block, two do not, and there is no room for 80 pairs of blocks
    assert _path(65536, 500, rows=(1, 80), guidance=False) == B.SJD_PATH_CLUSTER
    assert _path(65536, 500, rows=(1, 80), guidance=True) == B.SJD_PATH_STREAM


def test_tiles_only_when_forced():
    for V in (2048, 4096, 50176, 65536, 131072, 524288, 528384):
        for K in (1, 64, 2000, V // 2 + V // 16, V):
            for dtype in (B.SJD_BF16, B.SJD_F32):
                assert _path(V, K, dtype=dtype) != B.SJD_PATH_TILES, (V, K)


def test_refusals():
    with pytest.raises(B.SjdError):
        _path(65530, 10)
    with pytest.raises(B.SjdError):
        _path(65536, 0)
