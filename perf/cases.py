"""The work whose speed matters to a user of the library, as measurable cases.

Every case goes through the public binding (paper_2104_06800_gb300.voldor):
whole windows and batches as a visual-odometry front end runs them, and the
single steps, network passes and back-end calls a program drives by itself.
Inputs are seeded synthetic scenes ray cast on the GPU: a street, a room of
boxes or two walls, with Fisk-distributed flow noise and moving blobs.

listed() gives the named cases, draw(rng) one more of the same ranges,
prepare / run what a program holds and calls, work the bytes and operations a
pass cannot do without, exact the results in 64 bits from the definitions.
"""
import math
import random

import numpy as np
import torch

from paper_2104_06800_gb300 import voldor as V

DEV = "cuda"
SAMPLES = 64            # P3P samples per pose step (the library's default)
P0 = 1e-3               # outlier density, gamma, Z_EPS: the library's defaults
GAMMA = 0.95
Z_EPS = 1e-6
BASELINE = 0.25         # m, stereo
DEPTH = {"street": (2.0, 80.0), "boxes": (1.0, 40.0), "walls": (2.0, 10.0)}
MOTION = {"street": (1.0, 1.55), "boxes": (0.2, 0.45), "walls": (0.1, 0.2)}
ALPHA = {"street": 1.0, "boxes": 0.5, "walls": 0.5}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest window a program estimates in one call: every launch counts
        dict(name="window_small", kind="window", scene="walls", prior="none", W=160, H=120, N=3,
             K=64, iters=3),
        # one window of a street sequence, the size the front end is quoted on
        dict(name="window_street", kind="window", scene="street", prior="none", W=1216, H=368,
             N=6, K=128, iters=8),
        # an offline job or a server: RGB-D windows of mixed size and length at once
        dict(name="batch_rgbd", kind="batch", scene="boxes", count=12, shapes=0, K=64, iters=5),
        # the steps a program schedules itself: depth (rows and columns, without
        # and with a stereo prior, ragged sizes), rigidness, poses
        dict(name="depth_street", kind="depth", scene="street", prior="none", W=1216, H=368, N=6,
             K=128, iter=2, direction=2, alpha1=0.0),
        dict(name="depth_stereo_odd", kind="depth", scene="boxes", prior="stereo", W=509, H=383,
             N=5, K=64, iter=1, direction=1, alpha1=0.0),
        dict(name="estep_street", kind="estep", scene="street", prior="none", W=1216, H=368, N=6,
             direction=3, alpha1=0.0),
        dict(name="pose_boxes", kind="pose", scene="boxes", prior="none", W=640, H=480, N=5,
             iter=1),
        # dense scoring of given poses on a caller's points
        dict(name="score_poses", kind="score", n=300001, m=256),
        # the learned initialiser: inference, and the gradients of a training step
        dict(name="cnn_forward", kind="cnn", train=False, scene="boxes", W=640, H=480, N=6),
        dict(name="cnn_train", kind="cnn", train=True, scene="boxes", W=640, H=480, N=6),
        # the back end: two keyframes aligned, and what follows a window (the
        # visibility score of its frames and the covariance of its poses)
        dict(name="keyframe_align", kind="align", scene="street", W=1216, H=368, conf=True),
        dict(name="after_window", kind="after", scene="street", prior="none", W=1216, H=368, N=6),
    ]


def _size(rng, most=1216 * 480):
    """Image sizes from 96 x 72 to 1216 x 480 pixels, spread over their logarithm, odd ones too."""
    px = math.exp(rng.uniform(math.log(96 * 72), math.log(most)))
    aspect = rng.uniform(1.2, 3.2)
    W = min(1216, max(96, int(round(math.sqrt(px * aspect)))))
    return W, min(480, max(72, int(round(px / W))))


def draw(rng):
    kind = rng.choice(["window", "window", "batch", "depth", "depth", "estep", "pose", "score",
                       "cnn", "cnn", "align", "after"])
    W, H = _size(rng)
    N = rng.randint(2, 8)
    scene = rng.choice(["street", "boxes", "walls"])
    prior = rng.choice(["none", "stereo", "rgbd"])
    alpha1 = rng.choice([0.0, 0.0, round(rng.uniform(0.005, 0.05), 4)])
    if kind == "window":
        return dict(kind=kind, scene=scene, prior=prior, W=W, H=H, N=N, K=rng.randint(32, 128),
                    iters=rng.randint(2, 8))
    if kind == "batch":
        return dict(kind=kind, scene=scene, count=rng.randint(2, 8),
                    shapes=rng.randint(1, 10 ** 6), K=rng.choice([48, 64]), iters=rng.randint(2, 5))
    if kind == "depth":
        return dict(kind=kind, scene=scene, prior=prior, W=W, H=H, N=N, K=rng.randint(32, 160),
                    iter=rng.randint(0, 6), direction=rng.randint(0, 3), alpha1=alpha1)
    if kind == "estep":
        return dict(kind=kind, scene=scene, prior=prior, W=W, H=H, N=N,
                    direction=rng.randint(0, 3), alpha1=alpha1)
    if kind == "pose":
        return dict(kind=kind, scene=scene, prior=prior, W=W, H=H, N=N, iter=rng.randint(0, 6))
    if kind == "score":
        return dict(kind=kind, n=int(math.exp(rng.uniform(math.log(500), math.log(5e5)))),
                    m=int(math.exp(rng.uniform(math.log(4), math.log(600)))))
    if kind == "cnn":
        return dict(kind=kind, train=rng.random() < 0.5, scene=scene, W=W, H=H, N=N)
    if kind == "align":
        return dict(kind=kind, scene=scene, W=max(W, 320), H=max(H, 180), conf=rng.random() < 0.5)
    return dict(kind="after", scene=scene, prior=prior, W=W, H=H, N=N)


def _batch_windows(case):
    """(W, H, N) of every window of a batch case."""
    if case["shapes"] == 0:
        sizes = [(320, 240), (640, 480), (1216, 368)]
        return [(*sizes[i % 3], 3 + i % 6) for i in range(case["count"])]
    rng = random.Random(case["shapes"])
    return [(*_size(rng, 640 * 480), rng.randint(3, 8)) for _ in range(case["count"])]


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------
class _Draws:
    """Seeded random numbers: host scalars and device tensors."""

    def __init__(self, seed):
        self.host = np.random.default_rng(seed)
        self.dev = torch.Generator(device=DEV)
        self.dev.manual_seed(int(seed) & 0x7FFFFFFF)

    def rand(self, *shape):
        return torch.rand(*shape, generator=self.dev, device=DEV, dtype=torch.float64)

    def randn(self, *shape):
        return torch.randn(*shape, generator=self.dev, device=DEV, dtype=torch.float64)


def _rot(axis, angle):
    a = np.asarray(axis, np.float64)
    a = a / np.linalg.norm(a)
    k = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    return np.eye(3) + math.sin(angle) * k + (1 - math.cos(angle)) * (k @ k)


def _compose(A, B):
    return np.hstack([A[:, :3] @ B[:, :3], (A[:, :3] @ B[:, 3] + A[:, 3])[:, None]])


def _t(x):
    return torch.as_tensor(np.asarray(x, np.float64), device=DEV)


class _Scene:
    """Planes and boxes of one scene, its camera and its N + 1 poses."""

    def __init__(self, d, style, W, H, N):
        h = d.host
        self.W, self.H = W, H
        f = {"street": 720.0 / 1216.0, "boxes": 525.0 / 640.0, "walls": 0.75}[style] * W
        self.K = (f, f, W / 2.0, H / 2.0)
        planes, boxes = [], []
        if style == "walls":
            for s in (1, -1):
                n = _rot([0, 1, 0], s * math.radians(h.uniform(15, 35))) @ [0, 0, 1.0]
                planes.append((n, h.uniform(3, 6) * n[2]))
            planes.append(([0, 0, 1.0], 10.0))
        elif style == "street":
            planes += [([0, -1.0, 0], -1.65), ([0, 0, 1.0], 80.0)]
            xl, xr = h.uniform(6, 12), h.uniform(6, 12)
            planes += [([1.0, 0, 0], -xl), ([-1.0, 0, 0], -xr)]
            for _ in range(12):
                z = h.uniform(12, 60)
                x = -h.uniform(2.5, xl - 1) if h.uniform() < 0.5 else h.uniform(2.5, xr - 1)
                boxes.append(([x - 0.9, 0.15, z - 2], [x + 0.9, 1.65, z + 2]))
        else:
            planes += [([0, -1.0, 0], -1.5), ([0, 0, 1.0], 40.0)]
            for _ in range(20):
                x, z = h.uniform(-12, 12), h.uniform(3, 36)
                sx, sy, sz = h.uniform(0.5, 3.0, 3)
                boxes.append(([x - sx / 2, 1.5 - sy, z - sz / 2], [x + sx / 2, 1.5, z + sz / 2]))
        self.planes = planes
        self.lo = _t([b[0] for b in boxes]) if boxes else None
        self.hi = _t([b[1] for b in boxes]) if boxes else None
        tmin, tmax = MOTION[style]
        G = [np.hstack([np.eye(3), np.zeros((3, 1))])]
        for _ in range(N):
            if style == "walls":
                T = _rot(h.normal(size=3), math.radians(h.uniform(0.5, 2.0)))
                tau = h.normal(size=3)
                tau *= h.uniform(tmin, tmax) / np.linalg.norm(tau)
            else:
                T = _rot([0, 1, 0], math.radians(h.uniform(-1.5, 1.5)))
                tau = np.array([h.normal(0, 0.02), h.normal(0, 0.01), -h.uniform(tmin, tmax)])
            G.append(_compose(np.hstack([T, tau[:, None]]), G[-1]))
        self.G = np.stack(G)
        v, u = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float64),
                              torch.arange(W, device=DEV, dtype=torch.float64), indexing="ij")
        self.u, self.v = u, v
        fx, fy, cx, cy = self.K
        self.rays = torch.stack([(u - cx) / fx, (v - cy) / fy, torch.ones_like(u)], -1)

    def cast(self, G):
        """World points [H, W, 3] and depth [H, W] that the camera of pose G sees."""
        R, tau = _t(G[:, :3]), _t(G[:, 3])
        D, C = self.rays @ R, -(R.T @ tau)
        lam = torch.full_like(self.u, math.inf)
        for n, dist in self.planes:
            n = _t(n)
            l = (dist - n @ C) / (D @ n)
            lam = torch.minimum(lam, torch.where((l > 1e-6) & torch.isfinite(l), l, math.inf))
        if self.lo is not None:
            for lo, hi in zip(self.lo, self.hi):
                a, b = (lo - C) / D, (hi - C) / D
                near = torch.minimum(a, b).nan_to_num(nan=-math.inf).amax(-1)
                far = torch.maximum(a, b).nan_to_num(nan=math.inf).amin(-1)
                lam = torch.minimum(lam, torch.where((far >= near) & (near > 1e-6), near, math.inf))
        lam = torch.where(torch.isfinite(lam), lam, 1e3)
        return C + D * lam[..., None], lam

    def blobs(self, d, frac):
        """Ellipses that cover about `frac` of the image."""
        m = torch.zeros_like(self.u, dtype=torch.bool)
        r = max(6.0, self.W / 20.0)
        for _ in range(max(1, round(frac * self.W * self.H / (0.5 * r * r * math.pi)))):
            cu, cv = d.host.uniform(0, self.W), d.host.uniform(0, self.H)
            a, b = d.host.uniform(0.4 * r, 1.2 * r, 2)
            m |= ((self.u - cu) / a) ** 2 + ((self.v - cv) / b) ** 2 <= 1
        return m

    def flows(self, d, N, alpha, moving):
        """Noisy flows [N, H, W, 2] float32 and the masks of what moves by itself."""
        fx, fy, cx, cy = self.K
        out, masks = [], []
        for t in range(1, N + 1):
            P, _ = self.cast(self.G[t - 1])
            X = P @ _t(self.G[t][:, :3]).T + _t(self.G[t][:, 3])
            z = X[..., 2].clamp(min=1e-9)
            f = torch.stack([fx * X[..., 0] / z + cx - self.u, fy * X[..., 1] / z + cy - self.v], -1)
            f[X[..., 2] < 0.5] = 0.0
            m = self.blobs(d, moving)
            f[m] = _t(d.host.uniform(5, 30, 2) * d.host.choice([-1, 1], 2))
            r = d.rand(self.H, self.W).clamp(1e-9, 1 - 1e-9)
            mag, ang = alpha * torch.sqrt(r / (1 - r)), 2 * math.pi * d.rand(self.H, self.W)
            out.append(f + torch.stack([mag * torch.cos(ang), mag * torch.sin(ang)], -1))
            masks.append(m)
        return torch.stack(out).float().contiguous(), torch.stack(masks)


def _window(seed, style, prior, W, H, N):
    """One window's inputs: scene, flows, prior and inverse-depth range."""
    d = _Draws(seed)
    sc = _Scene(d, style, W, H, N)
    flow, moving = sc.flows(d, N, ALPHA[style], 0.05)
    Z = sc.cast(sc.G[0])[1]
    w = dict(d=d, scene=sc, W=W, H=H, N=N, K=sc.K, flow=flow, moving=moving, Z=Z, prior=prior,
             alpha0=ALPHA[style])
    holes = sc.blobs(d, 0.04) | (d.rand(H, W) < 0.04)
    if prior == "stereo":
        x = sc.K[0] * BASELINE / Z + 0.5 * d.randn(H, W)
        w["prior_map"] = torch.where(holes, math.nan, x).float()
    elif prior == "rgbd":
        w["prior_map"] = torch.where(holes, math.nan, Z * (1 + 0.01 * d.randn(H, W))).float()
    dmin, dmax = DEPTH[style]
    lo, hi = MOTION[style] if prior == "none" else (1.0, 1.0)
    w["range_free"] = float(np.float32(0.5 * lo / dmax)), float(np.float32(2.0 * hi / dmin))
    w["range_metric"] = float(np.float32(0.5 / dmax)), float(np.float32(2.0 / dmin))
    return w


def _mid_run_state(w):
    """A state as in the middle of a run, in metric units: inverse depth, rigidness, poses."""
    d, N, H, W = w["d"], w["N"], w["H"], w["W"]
    lo, hi = w["range_metric"]
    rho = (1 + 0.02 * d.randn(H, W)) / w["Z"]
    lost = d.rand(H, W) < 0.08
    rho = torch.where(lost, lo + (hi - lo) * d.rand(H, W), rho).clamp(lo, hi).float()
    q = torch.where(w["moving"], 0.3 * d.rand(N, H, W), 1 - 0.2 * d.rand(N, H, W)).float()
    qhat = (0.2 + 0.8 * d.rand(H, W)).float()
    G = w["scene"].G.copy()
    for t in range(1, N + 1):
        dR = _rot(d.host.normal(size=3), 5e-4)
        off = d.host.normal(size=3) * 0.003 * np.linalg.norm(G[t][:, 3])
        G[t] = _compose(np.hstack([dR, off[:, None]]), G[t])
    return rho, q, qhat, G


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
class _Owned:
    """A library handle that is destroyed with the state that holds it."""

    def __init__(self, handle, destroy):
        self.handle, self.destroy = handle, destroy

    def __del__(self):
        self.destroy(self.handle)


def _params(w, rng_name, K=64, alpha1=0.0, seed=1):
    lo, hi = w[rng_name]
    return V.vd_params_default(fisk_alpha0=w["alpha0"], fisk_alpha1=alpha1, outlier_density=P0,
                               gamma_stay=GAMMA, rho_min=lo, rho_max=hi, n_hyp=K,
                               n_pose_samples=SAMPLES, seed=seed)


def _push(ctx, w):
    for t in range(1, w["N"] + 1):
        V.vd_push_flow(ctx, t, w["flow"][t - 1])
    if w["prior"] == "stereo":
        V.vd_push_stereo_prior(ctx, w["prior_map"], BASELINE)
    elif w["prior"] == "rgbd":
        V.vd_push_depth_prior(ctx, w["prior_map"])


def _maps(w):
    H, W, N = w["H"], w["W"], w["N"]
    e = lambda *s: torch.empty(*s, device=DEV)  # noqa: E731
    return dict(rho=e(H, W), q=e(N, H, W), conf=e(H, W), qhat=e(H, W), rho_star=e(H, W),
                e_star=e(H, W))


def _score_inputs(case, seed):
    d = _Draws(seed)
    n, m = case["n"], case["m"]
    K = (720.0, 720.0, 608.0, 184.0)
    uv = d.rand(n, 2) * torch.tensor([1216.0, 368.0], device=DEV, dtype=torch.float64)
    Z = 2.0 * (80.0 / 2.0) ** d.rand(n)
    X = torch.stack([(uv[:, 0] - K[2]) / K[0] * Z, (uv[:, 1] - K[3]) / K[1] * Z, Z,
                     0.5 + 0.5 * d.rand(n)], -1).float()
    obs = torch.cat([uv + 0.7 * d.randn(n, 2), (0.5 + d.rand(n, 1)), torch.zeros_like(Z)[:, None]],
                    -1).float()
    poses = np.stack([np.hstack([_rot(d.host.normal(size=3), abs(d.host.normal()) * 2e-3),
                                 0.05 * d.host.normal(size=(3, 1))]) for _ in range(m)])
    return X.contiguous(), obs.contiguous(), _t(poses.reshape(m, 12)), _t(K)


def _cnn_layers(N):
    c0 = 16 if 2 * N + 4 <= 16 else 32
    return list(zip([c0, 32, 32, 32, 32, 32], [32, 32, 32, 32, 32, 1 + N]))


def _cnn_inputs(case, seed):
    w = _window(seed, case["scene"], "none", case["W"], case["H"], case["N"])
    h = w["d"].host
    parts = []
    for cin, cout in _cnn_layers(case["N"]):
        parts += [h.normal(size=cout * 9 * cin) * math.sqrt(2.0 / (9 * cin)),
                  0.01 * h.normal(size=cout)]
    w["theta"] = np.concatenate(parts).astype(np.float32)
    T1 = w["scene"].G[1].copy()
    scale = np.linalg.norm(T1[:, 3])
    T1[:, 3] /= scale
    w["T1"] = T1
    w["rho_t"] = (scale / w["Z"]).clamp(*w["range_free"]).float().contiguous()
    w["q_t"] = (~w["moving"]).float().contiguous()
    w["mask"] = (w["d"].rand(case["H"], case["W"]) < 0.9).to(torch.uint8)
    return w


def _align_inputs(case, seed):
    d = _Draws(seed)
    sc = _Scene(d, case["scene"], case["W"], case["H"], 2)
    maps = []
    for G in (sc.G[0], sc.G[2]):
        Z = sc.cast(G)[1]
        p = d.host.uniform(0, 2 * math.pi, 3)
        field = 0.002 * (torch.sin(sc.u / 97 + p[0]) + torch.sin(sc.v / 41 + p[1]) +
                         torch.sin((sc.u + sc.v) / 163 + p[2]))
        maps.append(torch.where(d.rand(sc.H, sc.W) < 0.02, math.nan, Z * (1 + field)).float())
    R, tau = sc.G[2][:, :3], sc.G[2][:, 3]
    T = np.hstack([R.T, (-R.T @ tau)[:, None]])
    off = d.host.normal(size=3)
    off *= 0.02 * np.linalg.norm(T[:, 3]) / np.linalg.norm(off)
    T0 = np.hstack([_rot(d.host.normal(size=3), 0.003) @ T[:, :3], (T[:, 3] + off)[:, None]])
    conf = (0.5 + 0.5 * d.rand(sc.H, sc.W)).float() if case["conf"] else None
    return dict(d1=maps[0], d2=maps[1], conf=conf, K=sc.K, T0=T0, s0=1.02, c=0.01)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "score":
        X, obs, poses, K = _score_inputs(case, seed)
        return dict(case=case, args=(X, obs, poses, K),
                    out=torch.empty(case["m"], device=DEV, dtype=torch.float64))
    if kind == "align":
        return dict(case=case, **_align_inputs(case, seed))
    if kind == "cnn":
        w = _cnn_inputs(case, seed)
        net = _Owned(V.vd_cnn_create(case["N"], 0), V.vd_cnn_destroy)
        V.vd_cnn_set_params(net.handle, w["theta"])
        return dict(case=case, net=net, w=w, out=_maps(w))
    if kind == "batch":
        ws = [_window(seed * 1000 + i, case["scene"], "rgbd", *s)
              for i, s in enumerate(_batch_windows(case))]
        b = _Owned(V.vd_batch_create([(w["W"], w["H"], w["N"], w["K"]) for w in ws],
                                     [_params(w, "range_free", case["K"], seed=1 + i)
                                      for i, w in enumerate(ws)]), V.vd_batch_destroy)
        return dict(case=case, batch=b, ws=ws, out=[_maps(w) for w in ws],
                    ctx=[V.vd_batch_window(b.handle, i) for i in range(len(ws))])
    w = _window(seed, case["scene"], case["prior"], case["W"], case["H"], case["N"])
    whole = kind == "window"
    p = _params(w, "range_free" if whole else "range_metric", case.get("K", 64),
                case.get("alpha1", 0.0))
    ctx = _Owned(V.vd_create(w["W"], w["H"], w["N"], w["K"], p), V.vd_destroy)
    st = dict(case=case, ctx=ctx, w=w, out=_maps(w))
    if not whole:
        _push(ctx.handle, w)
        st["rho"], st["q"], st["qhat"], st["G"] = _mid_run_state(w)
        V.vd_set_poses(ctx.handle, st["G"])
        V.vd_set_state(ctx.handle, st["rho"], st["q"], st["qhat"])
        if kind == "after":
            V.vd_pose_mstep(ctx.handle, 1, 0)
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "score":
        return V.vd_score_poses(*st["args"], 2.0, P0, st["out"])
    if kind == "align":
        r = V.vd_ka_align(st["d1"], st["d2"], st["K"], st["T0"], s0=st["s0"], conf2=st["conf"],
                          c=st["c"])
        return dict(T=r["T"], s=r["s"], cov=r["cov"], energy=r["energy"],
                    iterations=r["iterations"], n_valid=r["n_valid"])
    if kind == "cnn":
        w, o = st["w"], st["out"]
        geom = (w["K"], w["T1"])
        if case["train"]:
            # one step's gradients, as a loop takes them that averages over windows
            loss = V.vd_cnn_train_step(st["net"].handle, w["flow"], w["rho_t"], w["q_t"], w["mask"],
                                       *w["range_free"], 1.0, 1e-3, update=False, geom=geom)
            return dict(loss=loss, grads=V.vd_cnn_get_grads(st["net"].handle))
        V.vd_cnn_forward(st["net"].handle, w["flow"], *w["range_free"], o["rho"], o["q"], geom=geom)
        return dict(rho=o["rho"], q=o["q"])
    if kind == "batch":
        for c, w in zip(st["ctx"], st["ws"]):
            _push(c, w)
        V.vd_batch_run(st["batch"].handle, case["iters"], V.VD_BATCH_BOOTSTRAP, len(st["ws"]))
        return [dict(rho=V.vd_get_inv_depth(c, o["rho"]), q=V.vd_get_rigidness(c, o["q"]),
                     poses=V.vd_get_poses(c, w["N"]))
                for c, w, o in zip(st["ctx"], st["ws"], st["out"])]
    ctx, w, o = st["ctx"].handle, st["w"], st["out"]
    if kind == "window":
        _push(ctx, w)
        _, stats = V.vd_run_em(ctx, case["iters"])
        return dict(rho=V.vd_get_inv_depth(ctx, o["rho"]), q=V.vd_get_rigidness(ctx, o["q"]),
                    conf=V.vd_get_confidence(ctx, o["conf"]), poses=V.vd_get_poses(ctx, w["N"]),
                    energy=stats.mean_energy, rigid=stats.rigid_fraction)
    if kind == "depth":
        V.vd_set_state(ctx, st["rho"], st["q"], st["qhat"])
        V.vd_depth_mstep(ctx, case["iter"], case["direction"])
        V.vd_get_depth_candidates(ctx, o["rho_star"], o["e_star"])
        return dict(rho=V.vd_get_inv_depth(ctx, o["rho"]), rho_star=o["rho_star"],
                    e_star=o["e_star"])
    if kind == "estep":
        V.vd_rigidness_estep(ctx, case["direction"])
        r = dict(q=V.vd_get_rigidness(ctx, o["q"]), conf=V.vd_get_confidence(ctx, o["conf"]))
        if case["prior"] != "none":
            r["qhat"] = V.vd_get_prior_rigidness(ctx, o["qhat"])
        return r
    if kind == "pose":
        V.vd_set_poses(ctx, st["G"])
        V.vd_pose_mstep(ctx, case["iter"], 0)
        return V.vd_get_poses(ctx, w["N"])
    vc = V.vd_vc_scores(ctx)
    cov = V.vd_pose_covariance(ctx, w["N"])
    return dict(visible=np.array(vc["n_visible"]), covered=np.array(vc["n_covered"]),
                vc=np.array(vc["vc"]), mean=np.stack([c["mean"] for c in cov]),
                cov=np.stack([c["cov"] for c in cov]),
                inliers=np.array([c["n_inliers"] for c in cov]))


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _em_flops(px, N, K, iters):
    """A depth step takes every candidate's first term (17 operations, a fused
    multiply-add counted as two: 25) and the winner's others (37: 50); an
    E-step an emission and a smoothed posterior (80) per flow; a pose step one
    term (29) per rigid pixel and sample's best root."""
    return iters * px * (25.0 * K + 50.0 * (N - 1) + 80.0 * N + 29.0 * SAMPLES * N)


def work(case):
    kind = case["kind"]
    if kind == "score":
        return dict(bytes=32.0 * case["n"] + 104.0 * case["m"], flops=45.0 * case["n"] * case["m"])
    if kind == "batch":
        b = f = 0.0
        for W, H, N in _batch_windows(case):
            b += W * H * (8.0 * N + 4 + 4 * N + 4)
            f += _em_flops(W * H, N, case["K"], case["iters"])
        return dict(bytes=b, flops=f)
    px = float(case["W"] * case["H"])
    if kind == "align":
        return dict(bytes=px * (12 if case["conf"] else 8), flops=px * 200.0)
    N = case["N"]
    if kind == "cnn":
        mac = 9.0 * sum(ci * co for ci, co in _cnn_layers(N))
        if case["train"]:
            return dict(bytes=px * (8.0 * N + 4 + 4 * N + 1) + 8 * mac, flops=6 * mac * px)
        return dict(bytes=px * (8.0 * N + 4 + 4 * N) + 4 * mac, flops=2 * mac * px)
    p = 4.0 if case["prior"] != "none" else 0.0
    if kind == "window":
        return dict(bytes=px * (8.0 * N + p + 4 + 4 * N + 4),
                    flops=_em_flops(px, N, case["K"], case["iters"]))
    if kind == "depth":
        return dict(bytes=px * (12.0 * N + 4 + 2 * p + 12),
                    flops=px * (25.0 * case["K"] + 50.0 * (N - 1)))
    if kind == "estep":
        return dict(bytes=px * (8.0 * N + 4 + 2 * p + 4 * N + 4), flops=px * N * 80.0)
    if kind == "pose":
        return dict(bytes=px * (12.0 * N + 4), flops=px * N * 29.0 * SAMPLES)
    return dict(bytes=px * 4.0, flops=px * N * 25.0)


# ---------------------------------------------------------------------------
# the results in 64 bits, from the definitions
# ---------------------------------------------------------------------------
def _project64(w, G, rho, u, v):
    """Image position and camera depth of pixels (u, v) at inverse depth rho in the frame of pose G."""
    fx, fy, cx, cy = w["K"]
    rx, ry = (u - cx) / fx, (v - cy) / fy
    h = [G[r, 0] * rx + G[r, 1] * ry + G[r, 2] + rho * G[r, 3] for r in range(3)]
    return fx * h[0] / h[2] + cx, fy * h[1] / h[2] + cy, h[2]


def _bilinear64(F, x, y):
    H, W = F.shape[:2]
    x0, y0 = x.floor().clamp(0, W - 2).long(), y.floor().clamp(0, H - 2).long()
    ax, ay = (x - x0)[..., None], (y - y0)[..., None]
    top = F[y0, x0] + ax * (F[y0, x0 + 1] - F[y0, x0])
    bot = F[y0 + 1, x0] + ax * (F[y0 + 1, x0 + 1] - F[y0 + 1, x0])
    return top + ay * (bot - top)


def _terms64(w, G, rho, u, v, alpha1):
    """Per flow: observed, in front of camera t, and y = P0 / p1 of its residual."""
    H, W = w["H"], w["W"]
    xp, yp, front_prev = u, v, torch.ones_like(u, dtype=torch.bool)
    for t in range(w["N"]):
        F = w["flow64"][t]
        x, y, z = _project64(w, G[t + 1], rho, u, v)
        front = z > Z_EPS
        if t == 0:
            obs, f = front_prev, F[v.long(), u.long()]
        else:
            obs = front_prev & (xp >= 0) & (xp <= W - 1) & (yp >= 0) & (yp <= H - 1)
            f = _bilinear64(F, torch.where(obs, xp, 0.0), torch.where(obs, yp, 0.0))
        r2 = (f[..., 0] - (x - xp)) ** 2 + (f[..., 1] - (y - yp)) ** 2
        a2 = (w["alpha0"] + alpha1 * f.norm(dim=-1)) ** 2
        yield obs, front, P0 * math.pi * a2 * (1 + r2 / a2) ** 2
        xp, yp, front_prev = x, y, front


def _prior64(w, rho, u, v):
    """Where the pixels have a prior, and the ratio P0 / p1 (or uniform to Gaussian) of rho under it."""
    pv = w["prior_map"].double()[v.long(), u.long()]
    if w["prior"] == "stereo":
        ok = torch.isfinite(pv) & (pv > 0)
        a2 = w["alpha0"] ** 2
        r2 = (torch.where(ok, pv, 0.0) - w["K"][0] * BASELINE * rho) ** 2
        return ok, P0 * math.pi * a2 * (1 + r2 / a2) ** 2
    ok = torch.isfinite(pv) & (pv > 0)
    # the library keeps the prior's inverse depth in float32
    ph = (1.0 / torch.where(ok, pv, 1.0).float()).double()
    z = 0.5 * ((ph - rho) / (0.01 * ph)) ** 2 + math.log(math.sqrt(2 * math.pi) * 0.01 / 2.0)
    return ok, torch.exp(z)


def _energy64(w, S, rho, u, v, alpha1):
    E = torch.zeros_like(rho)
    ul, vl = u.long(), v.long()
    if w["prior"] != "none":
        ok, y = _prior64(w, rho, u, v)
        E = torch.where(ok, S["qhat"][vl, ul] * torch.where(torch.isfinite(y), torch.log1p(y),
                                                            y.log()), 0.0)
    for t, (obs, front, y) in enumerate(_terms64(w, S["G"], rho, u, v, alpha1)):
        l = torch.where(obs & front, torch.log1p(y), torch.where(obs, 64.0, 0.0))
        E = E + S["q"][t][vl, ul] * l
    return E


def _philox(j, it, block, seed):
    c = [j, torch.full_like(j, it), torch.zeros_like(j), torch.full_like(j, block)]
    k0, k1, m = seed & 0xFFFFFFFF, seed >> 32, 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((p1 >> 32) & m) ^ c[1] ^ k0, p1 & m, ((p0 >> 32) & m) ^ c[3] ^ k1, p0 & m]
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c


def _exact_depth(case, seed):
    w = _window(seed, case["scene"], case["prior"], case["W"], case["H"], case["N"])
    rho, q, qhat, G = _mid_run_state(w)
    W, H, K, a1 = w["W"], w["H"], case["K"], case["alpha1"]
    w["flow64"] = w["flow"].double()
    S = dict(q=q.double(), qhat=qhat.double(), G=_t(G))
    u, v = w["scene"].u, w["scene"].v
    lo, hi = (torch.tensor(x, device=DEV, dtype=torch.float32) for x in w["range_metric"])
    s = torch.tensor(max(0.5 * 2.0 ** -case["iter"], 1 / 64), device=DEV, dtype=torch.float32)
    two, one = (torch.tensor(x, device=DEV, dtype=torch.float32) for x in (2.0, 1.0))
    j = (v * W + u).long()
    prior = None
    if case["prior"] != "none":
        pv = w["prior_map"]
        ok = torch.isfinite(pv) & (pv > 0)
        if case["prior"] == "stereo":
            prior = pv / float(np.float32(w["K"][0] * BASELINE))
        else:
            prior = 1.0 / pv
        prior = torch.where(ok, prior.clamp(lo, hi), math.nan)
    best = rho.clamp(lo, hi)
    bestE = _energy64(w, S, best.double(), u, v, a1)
    for k in range(1, K):
        if (k - 1) % 4 == 0:
            words = _philox(j, case["iter"], (k - 1) // 4, 1)
        x = (words[(k - 1) % 4] >> 8).float() * 2.0 ** -24
        # float32 values, every operation rounded once
        c = lo + x * (hi - lo) if k <= (K - 1) // 2 else rho * (one + s * (two * x - one))
        c = c.clamp(lo, hi)
        if k == 1 and prior is not None:
            c = torch.where(torch.isnan(prior), c, prior)
        E = _energy64(w, S, c.double(), u, v, a1)
        take = E < bestE
        best, bestE = torch.where(take, c, best), torch.where(take, E, bestE)
    # propagation along the chains of the direction
    star, es, new = best.double(), bestE, best.double().clone()
    rows, rev = case["direction"] % 2 == 0, case["direction"] >= 2
    L = W if rows else H
    at = (lambda m: (slice(None), m)) if rows else (lambda m: (m, slice(None)))
    order = range(L - 1, -1, -1) if rev else range(L)
    cur = None
    for m in order:
        i = at(m)
        if cur is None:
            cur = star[i]
        else:
            cur = torch.where(_energy64(w, S, cur, u[i], v[i], a1) < es[i], cur, star[i])
        new[i] = cur
    return dict(rho=new, rho_star=star, e_star=es)


def _exact_estep(case, seed):
    w = _window(seed, case["scene"], case["prior"], case["W"], case["H"], case["N"])
    rho, _, _, G = _mid_run_state(w)
    w["flow64"] = w["flow"].double()
    u, v, r = w["scene"].u, w["scene"].v, rho.double()
    lam = torch.stack([torch.where(o & f, 1 / y, torch.where(o, 0.0, 1.0))
                       for o, f, y in _terms64(w, _t(G), r, u, v, case["alpha1"])])
    rows = case["direction"] % 2 == 0
    x = lam if rows else lam.transpose(1, 2)                  # chains along the last axis
    L, g = x.shape[-1], GAMMA
    a0, a1 = torch.ones_like(x), x.clone()
    for m in range(L):
        if m:
            a0[..., m] = g * a0[..., m - 1] + (1 - g) * a1[..., m - 1]
            a1[..., m] = ((1 - g) * a0[..., m - 1] + g * a1[..., m - 1]) * x[..., m]
        s = a0[..., m] + a1[..., m]
        a0[..., m] /= s
        a1[..., m] /= s
    b0, b1 = torch.ones_like(x[..., 0]), torch.ones_like(x[..., 0])
    q = torch.empty_like(x)
    for m in range(L - 1, -1, -1):
        q[..., m] = a1[..., m] * b1 / (a1[..., m] * b1 + a0[..., m] * b0)
        y1 = b1 * x[..., m]
        b0, b1 = g * b0 + (1 - g) * y1, (1 - g) * b0 + g * y1
        b0, b1 = b0 / (b0 + b1), b1 / (b0 + b1)
    q = q if rows else q.transpose(1, 2)
    out = dict(q=q.contiguous(), conf=q.sum(0) / w["N"])
    if case["prior"] != "none":
        ok, y = _prior64(w, r, u, v)
        out["qhat"] = torch.where(ok, 1 / (1 + y), 0.0)
        out["conf"] = (q.sum(0) + out["qhat"]) / (w["N"] + 1)
    return out


def _exact_score(case, seed):
    X, obs, poses, K = (x.double() for x in _score_inputs(case, seed))
    out = []
    for G in poses.reshape(-1, 3, 4):
        P = X[:, :3] @ G[:, :3].T + G[:, 3]
        z = torch.where(P[:, 2] > Z_EPS, P[:, 2], 1.0)
        r2 = (obs[:, 0] - K[0] * P[:, 0] / z - K[2]) ** 2 + (obs[:, 1] - K[1] * P[:, 1] / z - K[3]) ** 2
        a2 = obs[:, 2] ** 2
        l = torch.log1p(P0 * math.pi * a2 * (1 + r2 / a2) ** 2)
        out.append((X[:, 3] * torch.where(P[:, 2] > Z_EPS, l, 64.0)).sum())
    return torch.stack(out)


def _exact_cnn(case, seed):
    w = _cnn_inputs(case, seed)
    N, H, W = w["N"], w["H"], w["W"]
    theta = _t(w["theta"]).requires_grad_(case["train"])
    fx, fy, cx, cy = w["K"]
    T1, rays = _t(w["T1"]), w["scene"].rays
    h = rays @ T1[:, :3].T
    e = h + 0.1 * T1[:, 3]
    pos = lambda p: torch.stack([fx * p[..., 0] / p[..., 2] + cx, fy * p[..., 1] / p[..., 2] + cy])  # noqa: E731
    x0, x1 = pos(h), pos(e)
    here = torch.stack([w["scene"].u, w["scene"].v])
    ok = (h[..., 2] > 1e-6) & (e[..., 2] > 1e-6)
    geo = torch.where(ok, torch.cat([x0 - here, x1 - x0]), 0.0)
    layers = _cnn_layers(N)
    a = torch.zeros(1, layers[0][0], H, W, device=DEV, dtype=torch.float64)
    a[0, :2 * N] = w["flow"].double().permute(0, 3, 1, 2).reshape(2 * N, H, W) / 32
    a[0, 2 * N:2 * N + 4] = geo / 32
    at = 0
    for l, (cin, cout) in enumerate(layers):
        Wl = theta[at:at + cout * 9 * cin].reshape(cout, 3, 3, cin).permute(0, 3, 1, 2)
        at += cout * 9 * cin
        a = torch.nn.functional.conv2d(a, Wl, theta[at:at + cout], padding=1)
        at += cout
        if l < 5:
            a = a.relu()
    z, (lo, hi) = a[0], w["range_free"]
    if not case["train"]:
        return dict(rho=(math.sqrt(lo * hi) * z[0].exp()).clamp(lo, hi), q=z[1:].sigmoid())
    m = w["mask"].double()
    r = z[0] + 0.5 * math.log(lo * hi) - w["rho_t"].double().log()
    bce = torch.nn.functional.binary_cross_entropy_with_logits(z[1:], w["q_t"].double(),
                                                               reduction="none")
    loss = ((m * r * r).sum() + (m * bce).sum() / N) / m.sum()
    loss.backward()
    return dict(loss=float(loss), grads=theta.grad)


def _exact_align(case, seed):
    s = _align_inputs(case, seed)
    fx, fy, cx, cy = s["K"]
    th1, th2 = s["d1"].double(), s["d2"].double()
    H, W = th1.shape
    v, u = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float64),
                          torch.arange(W, device=DEV, dtype=torch.float64), indexing="ij")
    rays = torch.stack([(u - cx) / fx, (v - cy) / fy, torch.ones_like(u)], -1)
    good = lambda t: torch.isfinite(t) & (t > 0)  # noqa: E731
    P = th1[..., None] * rays
    dx, dy = P[1:-1, 2:] - P[1:-1, :-2], P[2:, 1:-1] - P[:-2, 1:-1]
    kx = (P[1:-1, 2:] - 2 * P[1:-1, 1:-1] + P[1:-1, :-2]).norm(dim=-1)
    ky = (P[2:, 1:-1] - 2 * P[1:-1, 1:-1] + P[:-2, 1:-1]).norm(dim=-1)
    c = torch.linalg.cross(dx, dy)
    g = good(th1)
    ok = (g[1:-1, 2:] & g[1:-1, :-2] & g[2:, 1:-1] & g[:-2, 1:-1] & g[1:-1, 1:-1] &
          (c.norm(dim=-1) > 0) & (kx <= 0.2 * dx.norm(dim=-1)) & (ky <= 0.2 * dy.norm(dim=-1)))
    c = c / c.norm(dim=-1, keepdim=True)
    c = torch.where((c * P[1:-1, 1:-1]).sum(-1, keepdim=True) > 0, -c, c)
    nrm = torch.zeros(H, W, 3, device=DEV, dtype=torch.float64)
    has = torch.zeros(H, W, device=DEV, dtype=torch.bool)
    nrm[1:-1, 1:-1], has[1:-1, 1:-1] = torch.where(ok[..., None], c, 0.0), ok
    g2 = good(th2)
    X2 = th2[g2][:, None] * rays[g2]
    C2 = s["conf"].double()[g2] if s["conf"] is not None else torch.ones_like(th2[g2])
    cc = s["c"]

    def evaluate(T, sc):
        Q = X2 @ _t(T[:, :3]).T + _t(T[:, 3])
        Z = Q[:, 2]
        x, y = fx * Q[:, 0] / Z + cx, fy * Q[:, 1] / Z + cy
        i = (Z > Z_EPS) & (x >= 0) & (x <= W - 1) & (y >= 0) & (y <= H - 1)
        Q, Z, x, y, C = Q[i], Z[i], x[i], y[i], C2[i]
        lu, lv = (x + 0.5).floor().long(), (y + 0.5).floor().long()
        D = sc * th1[lv, lu]
        i = has[lv, lu] & good(D) & ((Z - D).abs() <= 0.2 * D)
        Q, Z, D, C, lu, lv = Q[i], Z[i], D[i], C[i], lu[i], lv[i]
        n = nrm[lv, lu]
        A, B = (n * rays[lv, lu]).sum(-1), (n * Q).sum(-1)
        r = A / Z - B / (D * Z)
        wt = C / (1 + (r / cc) ** 2)
        J3 = -n / (D * Z)[:, None]
        J3[:, 2] += (B - A * D) / (D * Z * Z)
        J = torch.cat([torch.linalg.cross(Q, J3), J3, (B / (D * Z))[:, None]], -1)
        E = (C * 0.5 * cc * cc * torch.log1p((r / cc) ** 2)).sum()
        return (float(E), ((J * wt[:, None]).T @ J).cpu().numpy(), (J.T @ (wt * r)).cpu().numpy(),
                len(r))

    T, sc, lam, it = s["T0"].copy(), s["s0"], 1e-3, 0
    E, Hm, gr, n = evaluate(T, sc)
    while it < 50 and lam <= 1e10 and n > 0:
        it += 1
        dl = -np.linalg.solve(Hm + lam * np.diag(np.diag(Hm)), gr)
        th = np.linalg.norm(dl[:3])
        k = np.array([[0, -dl[2], dl[1]], [dl[2], 0, -dl[0]], [-dl[1], dl[0], 0]])
        small = th < 1e-4
        a = 1 - th * th / 6 if small else math.sin(th) / th
        b = 0.5 - th * th / 24 if small else (1 - math.cos(th)) / th ** 2
        d = 1 / 6 - th * th / 120 if small else (th - math.sin(th)) / th ** 3
        ex = np.hstack([np.eye(3) + a * k + b * k @ k,
                        ((np.eye(3) + b * k + d * k @ k) @ dl[3:6])[:, None]])
        Tn, sn = _compose(ex, T), sc * math.exp(dl[6])
        En, Hn, gn, nn = evaluate(Tn, sn)
        if nn > 0 and En < E:
            T, sc, E, Hm, gr, n = Tn, sn, En, Hn, gn, nn
            lam /= 10
        else:
            lam *= 10
        if np.linalg.norm(dl) < 1e-10:
            break
    return dict(T=T, s=float(sc), cov=np.linalg.inv(Hm)[:6, :6], energy=E, iterations=None,
                n_valid=None)


def exact(case, seed):
    """None for whole windows and pose steps: their poses are modes of a seeded
    Monte-Carlo posterior of the library's own solver, held to the bound of
    their type; and for the covariances, which start from such samples."""
    kind = case["kind"]
    if kind == "depth":
        return _exact_depth(case, seed)
    if kind == "estep":
        return _exact_estep(case, seed)
    if kind == "score":
        return _exact_score(case, seed)
    if kind == "cnn":
        return _exact_cnn(case, seed)
    if kind == "align":
        return _exact_align(case, seed)
    return None
