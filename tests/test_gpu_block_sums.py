"""The last block's FP64 sum over the blocks of a linearisation: one block, counts
beside its ten chains (9, 10, 11), beside the eighty partials that the chains
hold in flight (79, 80, 81, 160, 161), an odd count and the capacity of the
caller's-buffer form, with points that all differ, so that a block left out or
added twice shows.  Every form of the sums against the FP64 oracle."""
import ctypes

import numpy as np
import pytest

from helpers import I34, both_sides, compare_linearization
from test_gpu_hcache import CACHED
from test_zz_no_alloc import _close

pytestmark = pytest.mark.gpu

BLOCK = 128


@pytest.fixture(scope="module")
def glt():
    import paper_2607_16897_gb300 as g
    return g


def _scene(n, seed):
    """Noise images and n points on distinct sub-pixel positions, all usable."""
    W, H = 320, 240
    rng = np.random.default_rng(seed)
    ref, cur = (rng.integers(0, 256, size=(H, W), dtype=np.uint8) for _ in range(2))
    uvd = np.stack([rng.uniform(20, W - 20, n), rng.uniform(20, H - 20, n), rng.uniform(1, 4, n)], 1).astype(np.float32)
    return W, H, (200.0, 200.0, W / 2, H / 2), ref, cur, uvd


@pytest.mark.parametrize("blocks", [1, 2, 3, 9, 10, 11, 79, 80, 81, 157, 160, 161, 512])
def test_callers_buffers(glt, orc, blocks):
    import torch
    n = (blocks - 1) * BLOCK + (BLOCK if blocks == 512 else 1 + blocks % 5)
    W, H, K, ref, cur, uvd = _scene(n, blocks)
    o = orc.OracleTracker(W, H, K, levels=1)
    o.build_pyramid(0, ref)
    o.set_map_points(uvd)
    o.build_pyramid(1, cur)
    want = o.debug_linearize(0, I34, 0.02, 1.0, per_sample=False)
    assert want["n"] == 8 * n
    r, c, u = (torch.from_numpy(a).cuda() for a in (ref, cur, uvd))
    out = torch.full((46,), np.nan, dtype=torch.float64, device="cuda")
    T = (ctypes.c_double * 12)(*I34.ravel())
    rc = glt.glt_linearize_noalloc(r.data_ptr(), W, c.data_ptr(), W, W, H, 0, *K, u.data_ptr(), n, T, 0.02, 1.0, 9.0, 1e-3,
                                   out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert rc == glt.GLT_OK
    _close(out.cpu().numpy(), want, blocks)


@pytest.mark.parametrize("form", ["forward", "mixed", "cached"])
@pytest.mark.parametrize("blocks", [1, 3, 11, 81, 157])
def test_tracker(glt, orc, blocks, form):
    n = (blocks - 1) * BLOCK + 1 + blocks % 5
    W, H, K, ref, cur, uvd = _scene(n, 1000 + blocks)
    cfg = {"forward": {}, "mixed": dict(precision="mixed"), "cached": CACHED}[form]
    trk, o = both_sides(glt, orc, W, H, K, ref, cur, uvd, levels=1, **cfg)
    g, w = trk.debug_linearize(0, I34, 0.02, 1.0), o.debug_linearize(0, I34, 0.02, 1.0)
    assert w["n"] == 8 * n
    compare_linearization(g, w, f"{form} {blocks} blocks")
    trk.close()
