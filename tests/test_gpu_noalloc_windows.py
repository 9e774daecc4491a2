"""glt_linearize_noalloc on levels of any address and pitch: points over the
whole image, so that windows touch the level's first and last byte, give the
same FP64 sums bit for bit whatever the alignment, and the oracle's; and the
sum over an even, an odd and a single number of blocks."""
import ctypes

import numpy as np
import pytest

from test_zz_no_alloc import _close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,n", [(64, 48, 128), (331, 243, 129), (333, 241, 700), (16, 16, 256)])
def test_any_alignment(orc, W, H, n):
    import torch

    import paper_2607_16897_gb300 as glt
    rng = np.random.default_rng(W + n)
    ref, cur = (rng.integers(0, 256, size=(H, W), dtype=np.uint8) for _ in range(2))
    K = (200.0, 200.0, W / 2, H / 2)
    uvd = np.stack([rng.uniform(0, W, n), rng.uniform(0, H, n), rng.uniform(1, 4, n)], 1).astype(np.float32)
    # the corners of the usable range
    uvd[:4] = [[3, 3, 2], [W - 5, 3, 2], [3, H - 5, 2], [W - 5, H - 5, 2]]
    T = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, 0]], np.float64)
    uvd_dev = torch.from_numpy(uvd).cuda()
    out = torch.zeros(46, dtype=torch.float64, device="cuda")
    o = orc.OracleTracker(W, H, K, levels=1)
    o.build_pyramid(0, ref)
    o.set_map_points(uvd)
    o.build_pyramid(1, cur)
    want = o.debug_linearize(0, T, 0.02, 1.0, per_sample=False)
    first = None
    for extra, offset in ((0, 0), (1, 0), (3, 1), (4, 2), (13, 3), (8, 8)):
        bufs = []
        for img in (ref, cur):
            host = rng.integers(0, 256, size=offset + (W + extra) * (H - 1) + W, dtype=np.uint8)
            np.lib.stride_tricks.as_strided(host[offset:], (H, W), (W + extra, 1))[:] = img
            bufs.append(torch.from_numpy(host).cuda())
        rc = glt.glt_linearize_noalloc(bufs[0].data_ptr() + offset, W + extra, bufs[1].data_ptr() + offset, W + extra, W, H, 0,
                                       *K, uvd_dev.data_ptr(), n, T.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), 0.02, 1.0,
                                       9.0, 1e-3, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == glt.GLT_OK
        got = out.cpu().numpy()
        _close(got, want, (extra, offset))
        first = got if first is None else first
        assert np.array_equal(got, first), (extra, offset)
