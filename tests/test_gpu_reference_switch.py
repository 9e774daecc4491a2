"""A tracker whose reference changes: with the cached Hessian every new set of
map points brings a new H^-1, which the last of the blocks that sum H writes.
Two iterations a level, so that the pose still depends on H^-1 (a converged one
would not), over references of different images and point counts, none and
textureless ones between them, against the FP64 oracle set up anew for each."""
import numpy as np
import pytest

from helpers import I34, ROT_TOL, TRANS_TOL, pose_diff
from test_gpu_hcache import CACHED

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def glt():
    import paper_2607_16897_gb300 as g
    return g


# (seed of the pair, points; None: all of them on a reference without texture)
ORDERS = [[(1, 500), (2, 61), (3, 300), (1, 500)],
          [(4, 129), (4, 0), (5, 500), (5, None), (2, 128)],
          [(6, None), (6, 400), (7, 0), (7, 32)]]


@pytest.mark.parametrize("order", ORDERS, ids=["counts", "empty", "flat"])
@pytest.mark.parametrize("pattern", [0, 5, 7])
def test_every_reference_has_its_own_inverse(glt, orc, syn, pattern, order):
    cfg = dict(CACHED, levels=3, pattern=pattern, max_iters=[2, 2, 2])
    p = syn.pair_c1(order[0][0], sigma=2.0)
    W, H, K = p.cam.W, p.cam.H, p.cam.K
    trk = glt.Tracker(W, H, K, max_points=500, **cfg)
    statuses, poses = [], []
    for seed, n in order:
        p = syn.pair_c1(seed, sigma=2.0)
        ref = np.full_like(p.ref, 90) if n is None else p.ref
        uvd = p.uvd[:500 if n is None else n]
        o = orc.OracleTracker(W, H, K, **cfg)
        for t in (trk, o):
            t.build_pyramid(0, ref)
            t.set_map_points(uvd)
            t.build_pyramid(1, p.cur)
        g, r = trk.track_frame(I34, (0.05, 3.0)), o.track_frame(I34, (0.05, 3.0))
        ang, dt = pose_diff(g["T"], r["T"])
        assert ang <= ROT_TOL and dt <= TRANS_TOL, (seed, n, ang, dt)
        assert g["status"] == r["status"] and g["passes"] == r["passes"] and g["n_valid"] == r["n_valid"], (seed, n)
        statuses.append(g["status"])
        poses.append(np.linalg.norm(g["T"][:, 3]))
    trk.close()
    # the sequence does what it says: points move the pose, none and no texture do not
    for (seed, n), status, moved in zip(order, statuses, poses):
        want = glt.GLT_TRACK_NOT_PD if n is None else glt.GLT_TRACK_TOO_FEW_POINTS if n == 0 else 0
        assert status == want and (moved > 1e-3) == (want == 0), (seed, n, status, moved)
