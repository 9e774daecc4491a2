"""The work a user has this framework do, as cases that can be timed and compared.

Every case goes through the public binding (``Tracker``, ``Batch``, ``NN`` and the C entry points).  Frames are
rendered here: a camera in a textured box room (the room of the repository's benchmark, 8 x 3.2 x 9.5 m, sensor
noise sigma 2, a change of exposure), map points on the strongest gradient of each grid cell with their exact
depth, a start as far from the true pose as a constant-velocity prediction leaves it.

Kinds of case (``case["kind"]``):
  frame      one camera frame already on the device: pyramid and solve as one asynchronous call
  host       the same from a frame in pinned host memory, the result read back
  keyframe   a new reference frame and its map points, then the first frame tracked against them
  batch      many camera streams per step: one replay of the captured graph
  linearize  the normal equations of one pass on the caller's own device buffers
  train      a few steps of the proposal network's training, loss and weights back
  forward    the proposal network on a batch of inputs (its held-out evaluation)
"""
import ctypes
import math
import os
import tempfile

import numpy as np
import torch
import torch.nn.functional as F

import paper_2607_16897_gb300 as glt

DEV = "cuda"
ROOM_LO, ROOM_HI = (-4.0, -1.6, -3.0), (4.0, 1.6, 6.5)
TEXELS, TEXTURE_M = 1024, 8.0            # one wall texture: 8 x 8 m, repeated
PATTERN8 = ((0, 0), (-2, 0), (2, 0), (0, -2), (0, 2), (-1, -1), (1, -1), (-1, 1))
SIZES = ((320, 240), (640, 480), (752, 480), (1280, 720))
HUBER, ZMIN, MIN_VALID = 9.0, 1e-3, 16
LAMBDA0, LAMBDA_UP, LAMBDA_DOWN = 1e-4, 4.0, 0.5
EPS_STEP, EPS_STEP_COARSE, ACCEPT_STEP, MAX_ITERS = 1e-6, 3e-4, 1e-3, 10
NO_HUBER, ANY_STEP = 1e30, 1e30          # the paper's configuration: no robust weights, every step taken
LR, TRAINED_STEPS = 3e-4, 500
TRAINED = os.path.join(os.path.dirname(glt.__file__), "proposal_weights.npy")   # the weights it ships


def listed():
    return [
        # the smallest call: a 320 x 240 camera, few points (a drone's or headset's tracking camera)
        dict(name="frame_320x240", kind="frame", width=320, height=240, points=500, levels=3, pattern=0,
             precision="fp32", jacobian="forward", solve="fp64"),
        # the ordinary call: VGA, 2000 points, 4 levels (the benchmark's default workload)
        dict(name="frame_640x480", kind="frame", width=640, height=480, points=2000, levels=4, pattern=0,
             precision="fp32", jacobian="forward", solve="fp64"),
        # FP16 levels and a ragged size: an odd width, a number of points that fills no warp
        dict(name="frame_mixed_ragged", kind="frame", width=753, height=481, points=1337, levels=4, pattern=0,
             precision="mixed", jacobian="forward", solve="fp64"),
        # the largest single stream: 720p, 8000 points, 5 levels
        dict(name="frame_1280x720", kind="frame", width=1280, height=720, points=8000, levels=5, pattern=0,
             precision="fp32", jacobian="forward", solve="fp64"),
        # a per-frame caller with frames on the host
        dict(name="host_640x480", kind="host", width=640, height=480, points=2000, levels=4, pattern=0,
             precision="fp32", jacobian="forward", solve="fp64"),
        # the paper's own configuration: 7 x 7 patches, 6 levels, cached Hessian, plain Gauss-Newton
        dict(name="paper_640x480_7x7", kind="frame", width=640, height=480, points=2000, levels=6, pattern=7,
             precision="fp32", jacobian="ic", solve="fp64"),
        # the paper's larger one (11 x 11 at 752 x 480) on a keyframe: the reference side is built anew
        dict(name="keyframe_752x480_11x11", kind="keyframe", width=752, height=480, points=2000, levels=6,
             pattern=11, precision="fp32", jacobian="ic", solve="fp64"),
        # a server's batch: 64 cameras of mixed sizes and point counts, clusters sized by points
        dict(name="batch_64_mixed", kind="batch", streams=64, width=0, height=0, points=300, points_to=4000,
             levels=4, proposal=False, precision="fp32"),
        # 256 VGA cameras with the learned initial-pose proposal in front of the solve
        dict(name="batch_256_proposal", kind="batch", streams=256, width=640, height=480, points=2000,
             points_to=2000, levels=5, proposal=True, precision="fp32"),
        # one linearisation for a caller with its own solver and its own memory
        dict(name="linearize_20000", kind="linearize", width=1280, height=720, points=20000, level=0),
        # training of the proposal network, resumed from a checkpoint, with the batch its training script uses
        dict(name="train_256", kind="train", batch=256, steps=4),
        # its held-out evaluation: the validation pairs in one call
        dict(name="forward_5000", kind="forward", batch=5000),
    ]


def draw(rng):
    kind = rng.choice(("frame", "frame", "host", "frame", "keyframe", "batch", "linearize", "train", "forward"))
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    if kind in ("frame", "host", "keyframe"):
        w = log(320, 1280)
        h = max(240, min(720, int(w * rng.uniform(0.56, 0.76))))
        c = dict(kind=kind, width=w, height=h, points=log(300, 8000), levels=rng.randint(3, 5), pattern=0,
                 precision=rng.choice(("fp32", "fp32", "mixed")), jacobian=rng.choice(("forward", "forward", "ic")),
                 solve=rng.choice(("fp64", "fp64", "fp32")))
        if rng.random() < 0.3:
            # the paper's configuration: fewer points, each a whole patch; the coarsest level keeps 8 pixels
            c.update(points=log(300, 2000), levels=rng.randint(4, 5), pattern=rng.choice((5, 7, 11)),
                     precision="fp32", jacobian="ic", solve="fp64")
        return c
    if kind == "batch":
        proposal = rng.random() < 0.4
        lo = log(300, 2000)
        s = log(4, 128)
        w, h = rng.choice(SIZES + ((0, 0), (639, 477)))
        if proposal:
            w, h = 640, 480
        return dict(kind="batch", streams=s, width=w, height=h, points=lo, points_to=min(4000, 2 * lo),
                    levels=5 if proposal else rng.randint(3, 4), proposal=proposal,
                    precision="fp32" if proposal else rng.choice(("fp32", "fp32", "mixed")))
    if kind == "linearize":
        w = log(320, 1280)
        return dict(kind="linearize", width=w, height=int(w * 0.6), points=log(200, 60000), level=rng.randint(0, 2))
    if kind == "train":
        return dict(kind="train", batch=log(17, 256), steps=rng.randint(1, 4))
    return dict(kind="forward", batch=log(1, 5000))


# ---------------------------------------------------------------------------
# scene: poses, rendering, map points
# ---------------------------------------------------------------------------
def _focal(w):
    return 525.0 if w == 640 else 0.8 * w


def _rot(v):
    """Rotation matrix of a rotation vector (Rodrigues)."""
    th = float(np.linalg.norm(v))
    W = np.array([[0, -v[2], v[1]], [v[2], 0, -v[0]], [-v[1], v[0], 0]])
    if th < 1e-12:
        return np.eye(3) + W
    return np.eye(3) + math.sin(th) / th * W + (1 - math.cos(th)) / th ** 2 * (W @ W)


def _poses(rng):
    """Camera-to-world pose of the reference, the motion T_cr (reference to current camera), a start as a
    constant-velocity prediction gives it, and the last inter-frame motion."""
    T_wc = np.zeros((3, 4))
    T_wc[:, :3] = _rot(rng.normal(size=3) * np.array([0.1, 0.3, 0.05]))
    T_wc[:, 3] = rng.uniform([-1.5, -0.4, -1.0], [1.5, 0.4, 1.0])
    T = np.zeros((3, 4))
    d = rng.normal(size=3)
    T[:, :3] = _rot(d / np.linalg.norm(d) * math.radians(rng.uniform(0.3, 2.0)))
    d = rng.normal(size=3)
    T[:, 3] = d / np.linalg.norm(d) * rng.uniform(0.01, 0.06)
    T0 = T.copy()
    T0[:, :3] = T[:, :3] @ _rot(rng.normal(size=3) * math.radians(0.06))
    T0[:, 3] += rng.normal(size=3) * 1.5e-3
    M = np.zeros((3, 4))
    M[:, :3] = _rot(rng.normal(size=3) * math.radians(0.6))
    M[:, 3] = rng.normal(size=3) * 0.015
    return T_wc, T, T0, M


def _textures(gen):
    """Six periodic wall textures: band-limited noise, 0.5 to 16 cycles/m, amplitude falling with frequency."""
    k = torch.fft.fftfreq(TEXELS, device=DEV)[:, None] * TEXELS / TEXTURE_M
    l = torch.fft.rfftfreq(TEXELS, device=DEV)[None, :] * TEXELS / TEXTURE_M
    r = torch.sqrt(k * k + l * l)
    amp = torch.where((r >= 0.5) & (r <= 16.0), r.clamp(min=0.5) ** -1.6, torch.zeros_like(r))
    z = torch.randn(6, TEXELS, TEXELS, device=DEV, generator=gen)
    t = torch.fft.irfft2(torch.fft.rfft2(z) * amp, s=(TEXELS, TEXELS))
    t = t / t.std(dim=(1, 2), keepdim=True)
    return (125.0 + 38.0 * t).clamp(30.0, 220.0).reshape(6, -1)


def _cast(T_wc, K, u, v):
    """Depth, wall and the two wall coordinates (m) that each pixel's ray meets."""
    o = [float(T_wc[i, 3]) for i in range(3)]
    x, y = (u - K[2]) / K[0], (v - K[3]) / K[1]
    d = [float(T_wc[i, 0]) * x + float(T_wc[i, 1]) * y + float(T_wc[i, 2]) for i in range(3)]
    ts = [torch.where(d[i] > 0, ROOM_HI[i] - o[i], ROOM_LO[i] - o[i]) / torch.where(d[i].abs() < 1e-9, 1e-9, d[i])
          for i in range(3)]
    t = torch.minimum(torch.minimum(ts[0], ts[1]), ts[2])
    axis = torch.where(t == ts[0], 0, torch.where(t == ts[1], 1, 2))
    p = [o[i] + t * d[i] for i in range(3)]
    side = torch.where(axis == 0, d[0] > 0, torch.where(axis == 1, d[1] > 0, d[2] > 0))
    return t, axis * 2 + side, torch.where(axis == 0, p[1], p[0]), torch.where(axis == 2, p[1], p[2])


def _render(tex, T_wc, K, w, h, a, b, gen):
    """8-bit frame, its depth and its wall ids."""
    v, u = torch.meshgrid(torch.arange(h, device=DEV, dtype=torch.float32),
                          torch.arange(w, device=DEV, dtype=torch.float32), indexing="ij")
    depth, wall, s, t = _cast(T_wc, K, u, v)
    s, t = s * (TEXELS / TEXTURE_M), t * (TEXELS / TEXTURE_M)
    s0, t0 = torch.floor(s), torch.floor(t)
    fs, ft = s - s0, t - t0
    s0, t0 = s0.long(), t0.long()
    flat, base, m = tex.reshape(-1), wall.long() * (TEXELS * TEXELS), TEXELS - 1
    at = lambda i, j: flat[base + ((t0 + j) & m) * TEXELS + ((s0 + i) & m)]  # noqa: E731
    L = (1 - ft) * ((1 - fs) * at(0, 0) + fs * at(1, 0)) + ft * ((1 - fs) * at(0, 1) + fs * at(1, 1))
    L = math.exp(a) * L + b + 2.0 * torch.randn(h, w, device=DEV, generator=gen)
    return torch.floor(L + 0.5).clamp(0, 255).to(torch.uint8), depth, wall


def _points(img, wall, T_wc, K, n, gen):
    """n map points (u, v, depth): the strongest gradient of each cell of a grid, away from the room's edges, then
    random ones; sub-pixel positions with the depth cast there."""
    h, w = img.shape
    f = img.float()
    g = torch.zeros_like(f)
    g[1:-1, 1:-1] = (f[1:-1, 2:] - f[1:-1, :-2]).abs() + (f[2:, 1:-1] - f[:-2, 1:-1]).abs()
    m = 8
    ok = torch.zeros_like(wall, dtype=torch.bool)
    c = wall[m:-m, m:-m]
    ok[m:-m, m:-m] = ((wall[:-2 * m, :-2 * m] == c) & (wall[2 * m:, :-2 * m] == c) & (wall[:-2 * m, 2 * m:] == c)
                      & (wall[2 * m:, 2 * m:] == c))
    score = torch.where(ok, g + torch.rand(h, w, device=DEV, generator=gen), torch.zeros_like(g))
    cell = max(1, min(int(math.sqrt(w * h / n)), 64))
    best, at = F.max_pool2d(score[None], cell, return_indices=True)
    best, at = best.reshape(-1), at.reshape(-1)
    k = min(n, best.numel())
    first = at[torch.topk(best, k).indices]
    more = torch.topk((score.reshape(-1) > 0).float() + torch.rand(h * w, device=DEV, generator=gen), n).indices
    at = torch.cat([first, more])[:n]
    jitter = torch.rand(2, n, device=DEV, generator=gen, dtype=torch.float64) - 0.5
    u, v = (at % w).double() + jitter[0], (at // w).double() + jitter[1]
    u, v = u.float().double(), v.float().double()
    depth = _cast(T_wc, K, u, v)[0]
    return torch.stack([u, v, depth], 1).float().contiguous()


def _seeded(seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 7919 + 11)
    return np.random.default_rng([int(seed), 2607]), gen


def _scene(rng, gen, tex, w, h, n, affine=True):
    """One stream's reference and current frame, points, start, motion."""
    K = (_focal(w), _focal(w), w / 2.0, h / 2.0)
    T_wc, T, T0, M = _poses(rng)
    Ti = np.zeros((3, 4))
    Ti[:, :3], Ti[:, 3] = T[:, :3].T, -T[:, :3].T @ T[:, 3]
    T_cur = np.zeros((3, 4))
    T_cur[:, :3], T_cur[:, 3] = T_wc[:, :3] @ Ti[:, :3], T_wc[:, :3] @ Ti[:, 3] + T_wc[:, 3]
    a, b = (float(rng.uniform(-0.05, 0.05)), float(rng.uniform(-4, 4))) if affine else (0.0, 0.0)
    ref, _, wall = _render(tex, T_wc, K, w, h, 0.0, 0.0, gen)
    cur = _render(tex, T_cur, K, w, h, a, b, gen)[0]
    uvd = _points(ref, wall, T_wc, K, n, gen)
    init = np.zeros(14)
    init[:12] = T0.reshape(12)
    if affine:
        init[12], init[13] = a + 0.003 * rng.normal(), b + 0.3 * rng.normal()
    return dict(K=K, w=w, h=h, ref=ref, cur=cur, uvd=uvd, init=init, motion=M)


def _config(case):
    """Keyword arguments of a tracker for the case; the paper's own configuration where patches are asked for."""
    kw = dict(levels=case["levels"], max_points=case["points"], precision=case["precision"])
    if case.get("pattern", 0):
        kw.update(pattern=case["pattern"], jacobian="ic", hessian="cached", affine=0, huber_k=NO_HUBER, lambda0=0.0,
                  accept_step=ANY_STEP, eps_step=0.0, eps_step_coarse=0.0)
    else:
        kw.update(jacobian=case.get("jacobian", "forward"), solve=case.get("solve", "fp64"))
    return kw


def _one(case, seed):
    rng, gen = _seeded(seed)
    return _scene(rng, gen, _textures(gen), case["width"], case["height"], case["points"],
                  affine=not case.get("pattern", 0))


def _streams(case, seed):
    rng, gen = _seeded(seed)
    tex = _textures(gen)
    # sizes and point counts belong to the installed cameras, not to their frames: they do not follow the seed
    shape = np.random.default_rng(case["streams"] * 131 + case["points"])
    out = []
    for _ in range(case["streams"]):
        w, h = SIZES[shape.integers(len(SIZES))] if case["width"] == 0 else (case["width"], case["height"])
        n = int(shape.integers(case["points"], case["points_to"] + 1))
        out.append(_scene(rng, gen, tex, w, h, n))
    return out


def _result_views(buf):
    """The fields of a device buffer of glt_result records."""
    f = glt.RESULT_DTYPE.fields
    d, i = buf.view(torch.float64), buf.view(torch.int32)
    f8 = lambda k, m: d[:, f[k][1] // 8: f[k][1] // 8 + m]  # noqa: E731
    i4 = lambda k, m: i[:, f[k][1] // 4: f[k][1] // 4 + m]  # noqa: E731
    return {"T": f8("T", 12), "a": f8("a", 1), "b": f8("b", 1), "cost": f8("cost", 1), "n_valid": i4("n_valid", 1),
            "iters_total": i4("iters_total", 1), "iters": i4("iters", glt.MAX_LEVELS), "passes": i4("passes", 1),
            "status": i4("status", 1)}


# ---------------------------------------------------------------------------
# proposal network inputs
# ---------------------------------------------------------------------------
LAYERS = (("w1", (16, 1, 3, 3)), ("b1", (16,)), ("w2", (32, 16, 3, 3)), ("b2", (32,)), ("w3", (64, 32, 3, 3)),
          ("b3", (64,)), ("w4", (128, 1286)), ("b4", (128,)), ("w5", (8, 128)), ("b5", (8,)))


def _net_params(rng):
    """He-initialised weights and small biases, as a training run starts or a trained file holds."""
    out = []
    for _, shape in LAYERS:
        if len(shape) > 1:
            out.append(rng.normal(size=shape) * math.sqrt(2.0 / np.prod(shape[1:])))
        else:
            out.append(rng.normal(size=shape) * 0.01)
    return np.concatenate([o.reshape(-1) for o in out]).astype(np.float32)


def _net_data(rng, n):
    """Residual images (gray levels / 64), motions and targets."""
    x = torch.from_numpy((rng.integers(-40, 41, size=(n, 1200)) / 64.0).astype(np.float32)).to(DEV)
    m = torch.from_numpy(rng.normal(size=(n, 6)).astype(np.float32)).to(DEV)
    t = torch.from_numpy(rng.normal(size=(n, 8)).astype(np.float32)).to(DEV)
    return x, m, t


def _train_state(rng):
    """Weights and Adam moments in the midst of a training run."""
    w = _net_params(rng)
    m = (3e-3 * rng.normal(size=w.size)).astype(np.float32)
    v = (1e-4 * np.exp(rng.normal(size=w.size))).astype(np.float32)
    return w, m, v


def _resume(net, w, m, v):
    """Loads a checkpoint file of the weights and moments (the format that include/glt.h states)."""
    with tempfile.TemporaryDirectory() as d:
        path = os.path.join(d, "net.ckpt")
        with open(path, "wb") as f:
            f.write(b"GLTNNCK1" + np.array([w.size, TRAINED_STEPS], "<i4").tobytes())
            for a in (w, m, v):
                f.write(a.astype("<f4").tobytes())
        net.load(path)
    return net


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("frame", "host", "keyframe"):
        s = _one(case, seed)
        trk = glt.Tracker(s["w"], s["h"], s["K"], **_config(case))
        st = dict(kind=kind, trk=trk, **s)
        if kind == "keyframe":
            st["uvd_host"] = s["uvd"].cpu().numpy()   # map points come from the host's indirect pipeline
        else:
            trk.build_pyramid(glt.GLT_REF, s["ref"])
            trk.set_map_points(s["uvd"])
        if kind == "host":
            pinned = torch.empty(s["cur"].shape, dtype=torch.uint8, pin_memory=True)
            pinned.copy_(s["cur"])
            st.update(pinned=pinned, frame=pinned.numpy(), T0=s["init"][:12].reshape(3, 4).copy(),
                      ab0=(float(s["init"][12]), float(s["init"][13])))
        else:
            out = torch.zeros((1, glt.RESULT_BYTES), dtype=torch.uint8, device=DEV)
            st.update(init_dev=torch.from_numpy(s["init"]).to(DEV), out=out, views=_result_views(out))
        return st
    if kind == "batch":
        streams = _streams(case, seed)
        trks = [glt.Tracker(s["w"], s["h"], s["K"], levels=case["levels"], max_points=len(s["uvd"]),
                            precision=case["precision"]) for s in streams]
        for t, s in zip(trks, streams):
            t.build_pyramid(glt.GLT_REF, s["ref"])
            t.set_map_points(s["uvd"])
        batch = glt.Batch(trks)
        if case["width"] == 0 or case["points"] != case["points_to"]:
            batch.set_proportional(384, 128)     # clusters in proportion to each stream's points
        else:
            batch.set_shape(2, 128)             # what the autotuner settles on for equal VGA streams
        frames = [s["cur"] for s in streams]
        out = torch.zeros((len(trks), glt.RESULT_BYTES), dtype=torch.uint8, device=DEV)
        st = dict(kind=kind, trks=trks, batch=batch, frames=frames, out=out, views=_result_views(out),
                  ptrs=torch.tensor([f.data_ptr() for f in frames], dtype=torch.int64, device=DEV),
                  init_dev=torch.from_numpy(np.stack([s["init"] for s in streams])).to(DEV))
        if case["proposal"]:
            st["net"] = glt.NN(len(trks), np.load(TRAINED))
            st["motion"] = torch.from_numpy(np.stack([s["motion"].reshape(12) for s in streams])).to(DEV)
            batch.set_proposal(st["net"], st["motion"])
        torch.cuda.synchronize()
        side = torch.cuda.Stream()
        batch.capture(st["ptrs"], st["init_dev"], out, side)
        return st
    if kind == "linearize":
        s = _one(case, seed)
        l = case["level"]
        T = (ctypes.c_double * 12)(*s["init"][:12])
        # the caller's own pyramid levels
        ref, cur = _pyramid(s["ref"], l + 1)[l].to(torch.uint8), _pyramid(s["cur"], l + 1)[l].to(torch.uint8)
        out = torch.zeros(46, dtype=torch.float64, device=DEV)
        return dict(kind=kind, ref=ref, cur=cur, uvd=s["uvd"], out=out, T=T,
                    args=(s["w"], s["h"], l, *s["K"]), a=float(s["init"][12]), b=float(s["init"][13]))
    rng = np.random.default_rng([int(seed), 4])
    if kind == "train":
        sets = [_net_data(rng, case["batch"]) for _ in range(case["steps"])]
        return dict(kind=kind, net=_resume(glt.NN(case["batch"]), *_train_state(rng)), sets=sets, batch=case["batch"],
                    loss=torch.zeros(case["steps"], device=DEV))
    x, m, _ = _net_data(rng, case["batch"])
    return dict(kind=kind, net=glt.NN(case["batch"], _net_params(rng)), x=x, m=m, batch=case["batch"],
                y=torch.zeros((case["batch"], 8), device=DEV))


def run(st):
    kind = st["kind"]
    if kind == "frame":
        st["trk"].track_image_async(st["cur"], st["init_dev"], st["out"])
        return st["views"]
    if kind == "host":
        return st["trk"].track_image(st["frame"], st["T0"], st["ab0"])
    if kind == "keyframe":
        trk = st["trk"]
        trk.build_pyramid(glt.GLT_REF, st["ref"])
        trk.set_map_points(st["uvd_host"])
        trk.track_image_async(st["cur"], st["init_dev"], st["out"])
        return st["views"]
    if kind == "batch":
        st["batch"].replay()
        return st["views"]
    if kind == "linearize":
        ref, cur, uvd, (w, h, l, fx, fy, cx, cy) = st["ref"], st["cur"], st["uvd"], st["args"]
        rc = glt.glt_linearize_noalloc(ref.data_ptr(), ref.shape[1], cur.data_ptr(), cur.shape[1], w, h, l, fx, fy,
                                       cx, cy, uvd.data_ptr(), uvd.shape[0], st["T"], st["a"], st["b"], HUBER, ZMIN,
                                       st["out"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if rc != 0:
            raise RuntimeError(glt.glt_last_error())
        return st["out"]
    if kind == "train":
        net, B = st["net"], st["batch"]
        for k, (x, m, t) in enumerate(st["sets"]):
            net.train_step(x, m, t, B, LR, st["loss"][k:])
        return {"loss": st["loss"], "weights": net.get_params()}
    st["net"].forward(st["x"], st["m"], st["y"], st["batch"])
    return st["y"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _track_work(w, h, n, levels, pattern, refresh=False):
    """Bytes: the frame once, the points and their reference patches once per level, the result.  Operations: the
    blur of each level and, per level, the samples of the fewest passes a level needs (its start and two steps;
    the fixed count in the paper's configuration), 160 operations each (20 with the Hessian kept)."""
    k = pattern * pattern if pattern else 8
    passes, ops = (1 + MAX_ITERS, 20) if pattern else (3, 160)
    table = levels * n * k * (12 if pattern else 4)
    pix = sum((w >> l) * (h >> l) for l in range(1, levels))
    nbytes = w * h + 24 * n + table + 14 * 8 + glt.RESULT_BYTES
    flops = pix * 16 + levels * passes * n * k * ops
    if refresh:
        nbytes += w * h + 12 * n + table
        flops += pix * 16 + levels * n * k * (30 + 42)
    return nbytes, flops


def work(case):
    kind = case["kind"]
    if kind in ("frame", "host", "keyframe"):
        b, f = _track_work(case["width"], case["height"], case["points"], case["levels"], case.get("pattern", 0),
                           kind == "keyframe")
        return {"bytes": b, "flops": f}
    if kind == "batch":
        w, h = (case["width"], case["height"]) if case["width"] else (748, 480)    # the mean of the four sizes
        b, f = _track_work(w, h, (case["points"] + case["points_to"]) // 2, case["levels"], 0)
        if case["proposal"]:
            f += 1.9e6
        return {"bytes": case["streams"] * b + (400e3 if case["proposal"] else 0), "flops": case["streams"] * f}
    if kind == "linearize":
        w, h, n = case["width"] >> case["level"], case["height"] >> case["level"], case["points"]
        return {"bytes": min(2 * w * h, 2 * 64 * n) + 12 * n + 46 * 8, "flops": n * 8 * 180}
    per = 2 * (300 * 16 * 9 + 80 * 32 * 144 + 20 * 64 * 288 + 128 * 1286 + 8 * 128)
    if kind == "train":
        B, s = case["batch"], case["steps"]
        return {"bytes": s * (B * (1200 + 6 + 8) * 4 + 189064 * 4 * 6) + 189064 * 4, "flops": s * 3 * B * per}
    return {"bytes": case["batch"] * (1200 + 6 + 8) * 4 + 189064 * 2, "flops": case["batch"] * per}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def _pyramid(img, levels):
    """Levels as float64 images of whole numbers: 5-tap binomial, clamped edges, even samples, rounded half up."""
    out = [img.double()]
    wk = (1.0, 4.0, 6.0, 4.0, 1.0)
    for _ in range(1, levels):
        p = F.pad(out[-1][None, None], (2, 2, 2, 2), mode="replicate")[0, 0]
        h, w = out[-1].shape[0] // 2, out[-1].shape[1] // 2
        r = sum(wk[j] * p[j:j + 2 * h:2] for j in range(5))
        r = sum(wk[j] * r[:, j:j + 2 * w:2] for j in range(5))
        out.append(torch.floor((r + 128.0) / 256.0))
    return out


def _offsets(pattern):
    if pattern == 0:
        d = torch.tensor(PATTERN8, device=DEV)
        return d[:, 0], d[:, 1], 2
    h = (pattern - 1) // 2
    r = torch.arange(-h, h + 1, device=DEV)
    return r.repeat(pattern), r.repeat_interleave(pattern), h


def _sample(img, xb, yb, al, be, dx, dy, grad):
    """Bilinear intensity (and halved central differences) at the pattern's samples of each point."""
    h, w = img.shape
    flat = img.reshape(-1)
    base = (yb[:, None] + dy) * w + xb[:, None] + dx
    at = lambda o: flat[(base + o).clamp(0, h * w - 1)]  # noqa: E731
    w00, w10, w01, w11 = [x[:, None] for x in ((1 - al) * (1 - be), al * (1 - be), (1 - al) * be, al * be)]
    mix = lambda f: w00 * f(0) + w10 * f(1) + w01 * f(w) + w11 * f(w + 1)  # noqa: E731
    I = mix(at)
    if not grad:
        return I, None, None
    return I, 0.5 * mix(lambda o: at(o + 1) - at(o - 1)), 0.5 * mix(lambda o: at(o + w) - at(o - w))


class _Exact:
    """One stream's solve in 64 bits."""

    def __init__(self, s, levels, pattern=0, ic=False, cached=False, huber=HUBER):
        self.K, self.uvd, self.pattern, self.ic, self.cached, self.huber = s["K"], s["uvd"].double(), pattern, ic, cached, huber
        self.levels = levels
        self.cur = _pyramid(s["cur"], levels)
        self.off = _offsets(pattern)
        d = self.uvd[:, 2]
        self.m = torch.stack([(self.uvd[:, 0] - self.K[2]) / self.K[0], (self.uvd[:, 1] - self.K[3]) / self.K[1],
                              torch.ones_like(d)], 1)
        self.xr = self.m * d[:, None]
        dx, dy, hh = self.off
        self.ref = []
        for l, img in enumerate(_pyramid(s["ref"], levels)):
            U, V = self.uvd[:, 0] * 2.0 ** -l, self.uvd[:, 1] * 2.0 ** -l
            xb, yb = torch.floor(U), torch.floor(V)
            ok = self._inside(xb, yb, img.shape)
            I0, gx, gy = _sample(img, xb.long(), yb.long(), U - xb, V - yb, dx, dy, ic)
            self.ref.append((ok, I0, gx, gy))

    def _inside(self, xb, yb, shape):
        hh = self.off[2]
        return (xb >= 1 + hh) & (xb <= shape[1] - 3 - hh) & (yb >= 1 + hh) & (yb <= shape[0] - 3 - hh)

    def _rows(self, l, sel, gx, gy, n, z, R):
        """Pose columns of the selected points' Jacobian rows; n: normalised position, z: depth, R: rotation."""
        s = 2.0 ** -l
        fx, fy = self.K[0] * s / z, self.K[1] * s / z
        a0 = fx[:, None] * (R[0] - n[:, :1] * R[2])
        a1 = fy[:, None] * (R[1] - n[:, 1:2] * R[2])
        Jt = gx[:, :, None] * a0[:, None] + gy[:, :, None] * a1[:, None]
        return torch.cat([Jt, torch.cross(self.xr[sel][:, None].expand_as(Jt), Jt, dim=2)], 2)

    def linearize(self, l, T, a, b):
        """H (8 x 8), g, E, n at a state; zero affine parts and unit weights where the Hessian is kept."""
        Td = torch.from_numpy(np.ascontiguousarray(T)).to(DEV)
        xc = self.xr @ Td[:, :3].T + Td[:, 3]
        z = xc[:, 2]
        n = xc / z[:, None]
        s = 2.0 ** -l
        u = self.uvd[:, 0] * s + self.K[0] * s * (n[:, 0] - self.m[:, 0])
        v = self.uvd[:, 1] * s + self.K[1] * s * (n[:, 1] - self.m[:, 1])
        xb, yb = torch.floor(u), torch.floor(v)
        img = self.cur[l]
        ok, I0, rx, ry = self.ref[l]
        ok = ok & (z > ZMIN) & self._inside(xb, yb, img.shape)
        sel = ok.nonzero()[:, 0]
        dx, dy, _ = self.off
        I, gx, gy = _sample(img, xb[sel].long(), yb[sel].long(), (u - xb)[sel], (v - yb)[sel], dx, dy, not self.ic)
        ea = math.exp(a)
        r = I - ea * I0[sel] - b
        ar = r.abs()
        w = torch.where(ar <= self.huber, torch.ones_like(r), self.huber / ar.clamp(min=1e-300))
        rho = torch.where(ar <= self.huber, 0.5 * r * r, self.huber * (ar - 0.5 * self.huber))
        if self.ic:
            eye = torch.eye(3, dtype=torch.float64, device=DEV)
            J = self._rows(l, sel, ea * rx[sel], ea * ry[sel], self.m[sel], self.uvd[sel, 2], eye)
        else:
            J = self._rows(l, sel, gx, gy, n[sel], z[sel], Td[:, :3])
        J = torch.cat([J, -ea * I0[sel][..., None], -torch.ones_like(r)[..., None]], 2).reshape(-1, 8)
        wr, r = (w * r).reshape(-1), r.reshape(-1)
        H = (J * w.reshape(-1, 1)).T @ J
        out = torch.cat([H.reshape(-1), J.T @ wr, rho.sum()[None], rho.new_tensor([float(rho.numel())])]).cpu().numpy()
        return out[:64].reshape(8, 8), out[64:72], float(out[72]), int(out[73])

    def kept(self, l):
        """The reference's own normal matrix of a level (unit weights, no gain)."""
        ok, _, rx, ry = self.ref[l]
        J = self._rows(l, ok, rx[ok], ry[ok], self.m[ok], self.uvd[ok, 2],
                       torch.eye(3, dtype=torch.float64, device=DEV)).reshape(-1, 6)
        return (J.T @ J).cpu().numpy()

    def solve(self, init):
        T = np.array(init[:12]).reshape(3, 4)
        q0 = T[0, :3] / np.linalg.norm(T[0, :3])
        q1 = T[1, :3] - (T[1, :3] @ q0) * q0
        q1 = q1 / np.linalg.norm(q1)
        T[0, :3], T[1, :3], T[2, :3] = q0, q1, np.cross(q0, q1)
        a, b, cost = float(init[12]), float(init[13]), math.nan
        lam0, stop, coarse, take = (0.0, 0.0, 0.0, ANY_STEP) if self.cached else (LAMBDA0, EPS_STEP, EPS_STEP_COARSE, ACCEPT_STEP)
        for l in range(self.levels - 1, -1, -1):
            Hc = self.kept(l) if self.cached else None
            H, g, E, n = self.linearize(l, T, a, b)
            if n < MIN_VALID:
                continue
            lam, it, eps = lam0, 0, coarse if l > 0 else stop
            cost = E / n
            if not _definite(math.exp(2 * a) * Hc if self.cached else H):
                continue
            while True:
                if self.cached:
                    d = np.zeros(8)
                    d[:6] = -np.linalg.solve(math.exp(2 * a) * Hc, g[:6])
                else:
                    d = -np.linalg.solve(H + lam * np.diag(np.diag(H)), g)
                step = np.abs(d[:6]).max()
                Tn, an, bn = _compose(T, _exp(d[:6])), a + d[6], b + d[7]
                if step < eps and step < take:
                    T, a, b = Tn, an, bn
                    break
                H2, g2, E2, n2 = self.linearize(l, Tn, an, bn)
                it += 1
                good = n2 >= MIN_VALID and (E2 * n < E * n2 or step < take)
                lam *= LAMBDA_DOWN if good else LAMBDA_UP
                if good:
                    T, a, b, H, g, E, n = Tn, an, bn, H2, g2, E2, n2
                if it >= MAX_ITERS or step < eps:
                    break
            cost = E / n
        return T, a, b, cost


def _definite(H):
    return bool(np.linalg.eigvalsh(H)[0] > 0)


def _exp(d):
    """SE(3) exponential of (translation, rotation)."""
    w, v = d[3:], d[:3]
    th2 = float(w @ w)
    W = np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])
    if th2 < 1e-6:
        A, B, C = 1 - th2 / 6 + th2 ** 2 / 120, 0.5 - th2 / 24 + th2 ** 2 / 720, 1 / 6 - th2 / 120 + th2 ** 2 / 5040
    else:
        th = math.sqrt(th2)
        A, B, C = math.sin(th) / th, 2 * math.sin(th / 2) ** 2 / th2, (th - math.sin(th)) / (th2 * th)
    T = np.zeros((3, 4))
    T[:, :3] = np.eye(3) + A * W + B * (W @ W)
    T[:, 3] = v + B * (W @ v) + C * (W @ (W @ v))
    return T


def _compose(A, B):
    T = A[:, :3] @ B
    T[:, 3] += A[:, 3]
    return T


def _log(M):
    """(translation, rotation) whose exponential is M; motions of a few degrees."""
    R = M[:, :3]
    vee = np.array([R[2, 1] - R[1, 2], R[0, 2] - R[2, 0], R[1, 0] - R[0, 1]])
    sn, cs = 0.5 * np.linalg.norm(vee), 0.5 * (np.trace(R) - 1)
    th = math.atan2(sn, cs)
    w = vee * (0.5 if th < 1e-8 else th / (2 * sn))
    W = np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])
    k = 1 / 12 + th ** 2 / 720 if th < 1e-3 else (1 - th * math.sin(th) / (2 * (1 - math.cos(th)))) / th ** 2
    return np.concatenate([M[:, 3] - 0.5 * W @ M[:, 3] + k * W @ (W @ M[:, 3]), w])


def _split(params):
    """Named weights, rounded to bfloat16 as the network uses them, in 64 bits."""
    out, at = {}, 0
    for name, shape in LAYERS:
        k = int(np.prod(shape))
        out[name] = params[at:at + k].bfloat16().double().reshape(shape)
        at += k
    return out


def _net(p, x, m):
    h = x.reshape(-1, 1, 30, 40)
    for k in ("1", "2", "3"):
        h = torch.relu(F.conv2d(h, p["w" + k], p["b" + k], stride=2, padding=1))
    h = torch.relu(torch.cat([h.flatten(1), m], 1) @ p["w4"].T + p["b4"])
    return h @ p["w5"].T + p["b5"]


def _track_outputs(found):
    """Laid out as run()'s result; counts are decisions, not computed numbers."""
    none = {k: None for k in ("n_valid", "iters_total", "iters", "passes", "status")}
    return {"T": np.stack([f[0].reshape(12) for f in found]), "a": np.array([[f[1]] for f in found]),
            "b": np.array([[f[2]] for f in found]), "cost": np.array([[f[3]] for f in found]), **none}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("frame", "host", "keyframe"):
        s, p = _one(case, seed), case.get("pattern", 0)
        x = _Exact(s, case["levels"], p, ic=bool(p) or case["jacobian"] == "ic", cached=bool(p), huber=NO_HUBER if p else HUBER)
        r = x.solve(s["init"])
        if kind != "host":
            return _track_outputs([r])
        return {"T": r[0], "a": r[1], "b": r[2], "cost": r[3], "n_valid": None, "iters_total": None, "iters": None,
                "passes": None, "status": None}
    if kind == "batch":
        streams = _streams(case, seed)
        if case["proposal"]:
            p = _split(torch.from_numpy(np.load(TRAINED).astype(np.float32)).to(DEV))
            for s in streams:
                x = (_pyramid(s["cur"], 5)[4] - _pyramid(s["ref"], 5)[4]) / 64.0
                m = torch.from_numpy(_log(s["motion"]) / 0.02).to(DEV)
                y = _net(p, x.reshape(1, -1), m[None])[0].cpu().numpy()
                init = s["init"].copy()
                init[:12] = _compose(init[:12].reshape(3, 4), _exp(0.01 * y[:6])).reshape(12)
                init[12] += 0.01 * y[6]
                init[13] += y[7]
                s["init"] = init
        return _track_outputs([_Exact(s, case["levels"]).solve(s["init"]) for s in streams])
    if kind == "linearize":
        s = _one(case, seed)
        H, g, E, n = _Exact(s, case["level"] + 1).linearize(case["level"], s["init"][:12].reshape(3, 4),
                                                            float(s["init"][12]), float(s["init"][13]))
        return np.concatenate([H[np.triu_indices(8)], g, [E, n]])
    rng = np.random.default_rng([int(seed), 4])
    if kind == "train":
        sets = [_net_data(rng, case["batch"]) for _ in range(case["steps"])]
        w, m1, m2 = (torch.from_numpy(a).to(DEV).double() for a in _train_state(rng))
        losses = []
        for k, (x, mo, t) in enumerate(sets):
            p = {n: v.requires_grad_() for n, v in _split(w).items()}
            loss = 0.5 * ((_net(p, x.double(), mo.double()) - t.double()) ** 2).sum() / case["batch"]
            loss.backward()
            g = torch.cat([p[n].grad.reshape(-1) for n, _ in LAYERS])
            m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
            n = TRAINED_STEPS + k + 1
            w = w - LR * (m1 / (1 - 0.9 ** n)) / (torch.sqrt(m2 / (1 - 0.999 ** n)) + 1e-8)
            losses.append(float(loss.detach()))
        return {"loss": np.array(losses), "weights": w.cpu().numpy()}
    x, m, _ = _net_data(rng, case["batch"])
    w = _split(torch.from_numpy(_net_params(rng)).to(DEV))
    return _net(w, x.double(), m.double())
