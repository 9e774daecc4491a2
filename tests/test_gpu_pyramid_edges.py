"""The pyramid where a thread's 16 columns and 11 rows meet a border: sizes
around a multiple of 16 columns and of 8 rows, blocks' and warps' edges within
a row, and frames whose pitch or address allows 16-byte loads, 4-byte loads or
neither; every level exactly as the oracle's."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def glt():
    import paper_2607_16897_gb300 as g
    return g


@pytest.mark.parametrize("W,H", [(16, 16), (17, 19), (18, 23), (31, 33), (32, 40), (33, 41), (34, 47), (47, 25), (241, 57),
                                 (511, 66), (513, 65), (530, 24), (753, 481), (1041, 131)])
@pytest.mark.parametrize("extra,offset", [(0, 0), (16, 0), (3, 0), (4, 4), (0, 1), (5, 8), (16, 16)])
def test_sizes_pitches_and_addresses(glt, orc, W, H, extra, offset):
    import torch
    levels = max(l for l in range(1, 5) if (min(W, H) >> (l - 1)) >= 8)
    rng = np.random.default_rng(W * 1000 + H * 10 + extra + offset)
    img = rng.integers(0, 256, size=(H, W), dtype=np.uint8)
    pitch = W + extra
    # the frame ends with its last row's last column
    host = rng.integers(0, 256, size=offset + pitch * (H - 1) + W, dtype=np.uint8)
    np.lib.stride_tricks.as_strided(host[offset:], (H, W), (pitch, 1))[:] = img
    buf = torch.from_numpy(host).cuda()
    trk = glt.Tracker(W, H, (100.0, 100.0, W / 2, H / 2), levels=levels, max_points=8)
    rc = glt.load().glt_build_pyramid(trk.handle, glt.GLT_CUR, ctypes.c_void_p(buf.data_ptr() + offset), pitch, 1, None)
    assert rc == glt.GLT_OK
    for l, want in enumerate(orc.pyramid(img, levels)):
        np.testing.assert_array_equal(trk.get_pyramid(glt.GLT_CUR, l), want, err_msg=f"level {l}")
    trk.close()
