"""The reference tables of the p x p patches: every patch size, shared by four
threads or owned by one, on an odd-sized image with points up to its borders,
in the three forms that read them (cached Hessian, inverse compositional,
forward), against the oracle with the tolerances of the other linearisation
tests; and the reference Hessian summed over more points than its blocks have
threads."""
import numpy as np
import pytest

from helpers import I34, ROT_TOL, TRANS_TOL, both_sides, compare_linearization, pose_diff
from test_gpu_hcache import CACHED

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def glt():
    import paper_2607_16897_gb300 as g
    return g


def _pair(syn, seed, N):
    p = syn.pair_c1(seed, sigma=2.0, W=331, H=243, N=N)
    # and points from the middle to beyond every border
    rng = np.random.default_rng(seed)
    edge = np.stack([rng.uniform(-3, 334, 60), rng.uniform(-3, 246, 60), rng.uniform(1, 5, 60)], 1)
    return p, np.concatenate([p.uvd, edge]).astype(np.float32)


@pytest.mark.parametrize("form", ["cached", "ic", "forward"])
@pytest.mark.parametrize("pattern", [3, 5, 7, 9, 11])
def test_patch_sizes(glt, orc, syn, pattern, form):
    p, uvd = _pair(syn, pattern, 217)
    cfg = dict(CACHED, pattern=pattern) if form == "cached" else dict(pattern=pattern, jacobian=form, affine=False)
    trk, o = both_sides(glt, orc, p.cam.W, p.cam.H, p.cam.K, p.ref, p.cur, uvd, levels=3, **cfg)
    T = orc.se3_exp(np.array([0.01, -0.02, 0.015, 0.004, -0.006, 0.003]))
    for level in range(3):
        compare_linearization(trk.debug_linearize(level, T, 0.02, 1.0), o.debug_linearize(level, T, 0.02, 1.0),
                              f"{form} {pattern} level {level}")
    g, r = trk.track_frame(I34, (0.05, 3.0)), o.track_frame(I34, (0.05, 3.0))
    ang, dt = pose_diff(g["T"], r["T"])
    assert ang <= ROT_TOL and dt <= TRANS_TOL, (ang, dt)
    assert g["status"] == r["status"] and g["n_valid"] == r["n_valid"]
    trk.close()


@pytest.mark.parametrize("pattern", [0, 7])
def test_reference_hessian_over_many_points(glt, orc, syn, pattern):
    p = syn.pair_c1(1, sigma=2.0, N=500)
    uvd = np.tile(p.uvd, (19, 1))[:9001]        # no multiple of the blocks' threads
    trk, o = both_sides(glt, orc, p.cam.W, p.cam.H, p.cam.K, p.ref, p.cur, uvd, levels=2, **dict(CACHED, pattern=pattern))
    for level in range(2):
        for _ in range(2):                      # the tickets start over for every reference
            g, r = trk.debug_linearize(level, I34, 0.0, 0.0), o.debug_linearize(level, I34, 0.0, 0.0)
            assert np.linalg.norm(g["H"] - r["H"]) <= 1e-5 * np.linalg.norm(r["H"])
            trk.set_map_points(uvd)
    trk.close()
