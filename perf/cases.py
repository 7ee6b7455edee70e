"""The work that users of this library have it do, as cases that can be timed and checked.

A case is one call pattern of the public API (Tracker, Batch, track_frame) at one size. Inputs are made from a seed
alone: a tilted textured plane seen from two nearby camera poses, with sensor noise and analytic normals, the
texture in pixels of the image so that every size tracks the same kind of frame. Strengths are the workloads' own
(the paper's leaf strengths with the pose prior 0.05 of the realistic sequences); frames that are differentiated take
a weaker photometric one, under which the derivative of many unrolled sweeps stays bounded.

One pass is one frame (a target frame with its sweeps, the pose, the inverse depth), or one frame and its backward
pass. Trackers keep their state from pass to pass as they do in a sequence, which is under way when the first pass
begins: prepare() has set the keyframe and tracked one target. Passes take two target frames in turn.
FP32 trackers return their pose and inverse depth in FP32, the precision of the state whose means they are.
"""
import math
import random

import numpy as np
import torch

import paper_2606_03989_gb300 as pv

STATE_VALUES = 151          # values of a pixel's state (mean, belief marginals, messages)
NODE_VALUES = 162           # values of a quadtree node's state
FLOPS_GRID = 5500           # arithmetic of one pixel update with four identity messages
FLOPS_TREE = 5000           # one identity message per pixel, and a third of a node with five
FLOPS_BACK = 4 * FLOPS_GRID  # the reverse pass of one pixel update

STRENGTHS = {"sigma_D": 5e-3, "sigma_P": 0.05, "sigma_R": 4e-4, "sigma_N": 1e-3, "sigma_Z": 1.0}
SIGMA_D_ADJOINT = 0.1
FIRST_SWEEPS = 20           # of the target that prepare() tracks
T_HUBER, DAMPING = 400.0, 0.5
NOISE, NOISE_ADJOINT = 0.25 / 255, 2.0 / 255  # of the intensities, whose range is [0, 1], at 256 pixels a row
RESOLUTIONS = ((128, 96), (256, 256), (320, 240), (640, 480))  # the batched workload's


def _track(name, width, height, iters, topology="grid", precision=32, kf_interval=0, host=False):
    c = {"kind": "track", "width": width, "height": height, "iters": iters, "topology": topology,
         "precision": precision, "kf_interval": kf_interval, "host": host}
    return dict(c, name=name) if name else c


def _batch(name, n, mix, iters, topology="grid", schedule="default"):
    c = {"kind": "batch", "n": n, "mix": mix, "iters": iters, "topology": topology, "schedule": schedule}
    return dict(c, name=name) if name else c


def _adjoint(name, width, height, iters, every, window):
    c = {"kind": "adjoint", "width": width, "height": height, "iters": iters, "every": every, "window": window}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the tiny pair: the smallest frame, where latency and launches count
        _track("tiny_64x48", 64, 48, 10),
        # a short-baseline sequence that re-anchors its keyframe at every frame, at a small sensor's size
        _track("anchor_128x96", 128, 96, 5, kf_interval=1),
        # the SCAMP-like sensor: 256x256, 20 sweeps per frame
        _track("room_256x256", 256, 256, 20),
        # a cropped camera image: no side a multiple of a tile's
        _track("ragged_333x251", 333, 251, 20),
        # the headline: a VGA frame from pinned host memory in, its pose back on the host
        _track("host_640x480", 640, 480, 20, host=True),
        # a 3 Mpx camera, the largest frame
        _track("large_2048x1536", 2048, 1536, 10),
        # the paper's hierarchical topology on a VGA frame
        _track("quadtree_640x480", 640, 480, 20, topology="quadtree"),
        # many sequences of the batched workload's resolutions at once, as a Batch runs them unless told otherwise
        _batch("batch_24", 24, 7, 20),
        # quadtree sequences in a batch
        _batch("batch_quadtree_12", 12, 5, 10, topology="quadtree"),
        # a frame differentiated through all of its 30 sweeps, every state kept (the adjoint workload's size)
        _adjoint("adjoint_320x240", 320, 240, 30, 1, 0),
        # a small frame differentiated over its last sweeps, states recomputed from checkpoints
        _adjoint("adjoint_window_160x120", 160, 120, 20, 5, 8),
        # FP64 verification of a small frame
        _track("fp64_128x96", 128, 96, 5, precision=64),
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    k = rng.random()
    if k < 0.55:
        width = _log_size(rng, 40, 2048)
        height = max(24, int(width * rng.uniform(0.6, 1.0)))
        iters = rng.choice((5, 10, 20))
        while width * height * iters > 2048 * 1536 * 10:
            iters //= 2
        precision, topology = 32, "grid"
        if rng.random() < 0.12 and width * height <= 160 * 160:
            precision, iters = 64, 5
        elif rng.random() < 0.3:
            topology = "quadtree"
        host = precision == 32 and rng.random() < 0.3
        kf = 1 if not host and topology == "grid" and precision == 32 and rng.random() < 0.2 else 0
        return _track(None, width, height, iters, topology, precision, kf, host)
    if k < 0.8:
        tree = rng.random() < 0.4
        return _batch(None, rng.randint(2, 12 if tree else 24), rng.randrange(1000), rng.choice((5, 10)),
                      "quadtree" if tree else "grid", "default" if tree else rng.choice(("default", "batched")))
    width = _log_size(rng, 48, 320)
    height = max(32, int(width * rng.uniform(0.6, 0.8)))
    iters = rng.choice((5, 10, 20))
    return _adjoint(None, width, height, iters, rng.choice((1, 5)), rng.choice((0, 0, 4)))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _camera(width, height):
    f = 0.8203 * width
    return (f, f, (width - 1) / 2.0, (height - 1) / 2.0, width, height)


def _pixel_grid(width, height, dev):
    v, u = torch.meshgrid(torch.arange(height, dtype=torch.float64, device=dev),
                          torch.arange(width, dtype=torch.float64, device=dev), indexing="ij")
    return u, v


def _scene(width, height, seed, noise, n_targets, dev):
    """Keyframe, target frames, keyframe normals (float32) and the keyframe's inverse depth (float64): a textured plane
    seen after motions of about a pixel and a half of image flow."""
    r = random.Random(seed)
    g = torch.Generator(device=dev).manual_seed(seed)
    fx, fy, cx, cy, _, _ = _camera(width, height)
    u, v = _pixel_grid(width, height, dev)
    x, y = (u - cx) / fx, (v - cy) / fy
    a, b, z0 = r.uniform(-0.3, 0.3), r.uniform(-0.3, 0.3), r.uniform(0.8, 1.3)
    z = z0 / (1 - a * x - b * y)
    nrm = math.sqrt(a * a + b * b + 1)
    normals = torch.stack([torch.full_like(x, a / nrm), torch.full_like(x, b / nrm), torch.full_like(x, -1 / nrm)], -1)
    # a larger image shows the same scene at more pixels: an upsampled frame, as the paper tracks them, whose motion
    # and wavelengths grow with it and whose noise per pixel falls
    scale = max(1.0, width / 256.0)
    waves = [(scale * math.exp(r.uniform(math.log(24.0), math.log(96.0))), r.uniform(0, 2 * math.pi), r.uniform(0, 2 * math.pi))
             for _ in range(6)]

    def texture(p, q):
        s = torch.full_like(p, 0.5)
        for lam, ang, ph in waves:
            k = 2 * math.pi / lam
            s = s + (0.5 / 6) * torch.sin(k * (math.cos(ang) * p + math.sin(ang) * q) + ph)
        return s

    def sensor(img):
        return (img + noise / scale * torch.randn(img.shape, generator=g, device=dev, dtype=torch.float64)).float().contiguous()

    def direction(size):
        d = [r.gauss(0, 1) for _ in range(3)]
        n = math.sqrt(sum(c * c for c in d))
        return [c / n * size for c in d]

    def motion():
        w = direction(0.5 * scale / fx)
        t = direction(1.2 * scale * z0 / fx)
        X = torch.stack([x * z, y * z, z], -1)
        Xt = X + torch.cross(torch.tensor(w, dtype=torch.float64, device=dev).expand_as(X), X, dim=-1)
        Xt = Xt + torch.tensor(t, dtype=torch.float64, device=dev)
        return fx * Xt[..., 0] / Xt[..., 2] + cx, fy * Xt[..., 1] / Xt[..., 2] + cy

    key = sensor(texture(u, v))
    targets = []
    for _ in range(n_targets):  # the first-order inverse flow is exact to the motion's square, far below the noise
        ut, vt = motion()
        targets.append(sensor(texture(2 * u - ut, 2 * v - vt)))
    return key, targets, normals.float().contiguous(), 1.0 / z


def _strengths(case):
    return dict(STRENGTHS, sigma_D=SIGMA_D_ADJOINT) if case["kind"] == "adjoint" else STRENGTHS


def _params(case):
    return pv.params(t_huber=T_HUBER, damping=DAMPING, kf_interval=case.get("kf_interval", 0),
                     precision=case.get("precision", 32), topology=1 if _tree(case) else 0, **_strengths(case))


def _tree(case):
    return case.get("topology") == "quadtree"


def _mix(case):
    """Sizes of a batch's sequences: the batched workload's resolutions, every fourth one a ragged crop."""
    r = random.Random(case["mix"])
    sizes = []
    for i in range(case["n"]):
        w, h = r.choice(RESOLUTIONS)
        sizes.append((w - r.randint(1, 40), h - r.randint(1, 40)) if i % 4 == 3 else (w, h))
    return sizes


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "batch":
        sizes = _mix(case)
        scenes = [_scene(w, h, seed * 1009 + i, NOISE, 2, dev) for i, (w, h) in enumerate(sizes)]
        batch = pv.Batch([_camera(w, h) for w, h in sizes], _params(case), dev)
        if case["schedule"] == "batched":
            batch.set_schedule(pv.SCHED_BATCHED)
        normals = [s[2] for s in scenes]
        frames = [[s[1][k] for s in scenes] for k in range(2)]
        for first in ([s[0] for s in scenes], frames[0]):
            batch.set_inputs(first, normals)
            batch.track(FIRST_SWEEPS)
        return {"case": case, "batch": batch, "frames": frames, "normals": normals, "pass": 1}
    adjoint = case["kind"] == "adjoint"
    w, h = case["width"], case["height"]
    key, targets, normals, inv = _scene(w, h, seed, NOISE_ADJOINT if adjoint else NOISE, 2, dev)
    trk = pv.Tracker(_camera(w, h), _params(case), dev)
    trk.track(key, normals)
    trk.track(targets[0], normals if case.get("kf_interval") else None, FIRST_SWEEPS)
    state = {"case": case, "trk": trk, "targets": targets, "normals": normals, "pass": 1}
    if adjoint:
        trk.set_recording(case["iters"], case["every"])
        trk.set_backward_window(case["window"])
        state["inv"] = inv
        state["sigmas"] = [torch.tensor(getattr(trk.params, s), dtype=torch.float32, requires_grad=True)
                           for s in ("sigma_D", "sigma_N")]
        state["key"] = key.requires_grad_(True)
        state["targets"] = [t.requires_grad_(True) for t in targets]
    elif case["host"]:
        state["targets"] = [t.cpu().pin_memory() for t in targets]
    return state


def _loss(xi, inv, inv_true):
    """A pose and an inverse-depth term, as a learned sensor setting would be trained on."""
    return (xi * xi).sum() + ((inv - inv_true) ** 2).mean()


def run(state):
    case, k = state["case"], state["pass"]
    state["pass"] = k + 1
    if case["kind"] == "batch":
        batch = state["batch"]
        batch.set_inputs(state["frames"][k % 2], state["normals"])
        batch.track(case["iters"])
        return {"poses": batch.poses().astype(np.float32)}
    trk = state["trk"]
    if case["kind"] == "adjoint":
        frame, key, (sigma_D, sigma_N) = state["targets"][k % 2], state["key"], state["sigmas"]
        xi, inv = pv.track_frame(trk, frame, key, sigma_D, sigma_N, case["iters"])
        grads = torch.autograd.grad(_loss(xi, inv, state["inv"]), [key, frame, sigma_D, sigma_N])
        return {"xi": xi.detach().float(), "inv_depth": inv.detach().float(),
                "d_key": grads[0], "d_frame": grads[1], "d_sigma_D": grads[2], "d_sigma_N": grads[3]}
    if case["host"]:
        trk.track_host(state["targets"][k % 2], None, case["iters"])
        return {"xi": trk.pose().astype(np.float32), "inv_depth": trk.inv_depth()}
    # an anchoring tracker takes the target as its next keyframe
    trk.track(state["targets"][k % 2], state["normals"] if case["kf_interval"] else None, case["iters"])
    xi = trk.pose_device()
    return {"xi": xi if case["precision"] == 64 else xi.float(), "inv_depth": trk.inv_depth()}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _nodes(w, h):
    n = 0
    while w > 1 or h > 1:
        w, h = (w + 1) // 2, (h + 1) // 2
        n += w * h
    return n


def work(case):
    """Bytes: the frame and the edge measurements read, the state carried from frame to frame read and written once,
    the results written; a differentiated frame also reads and writes its adjoint state. Flops: the pixel updates."""
    size = 8 if case.get("precision") == 64 else 4
    sizes = _mix(case) if case["kind"] == "batch" else [(case["width"], case["height"])]
    px = sum(w * h for w, h in sizes)
    values = px * STATE_VALUES
    if _tree(case):
        values += sum(_nodes(w, h) for w, h in sizes) * NODE_VALUES
    b = 2 * values * size + px * (4 + 4 * size)
    fl = px * case["iters"] * (FLOPS_TREE if _tree(case) else FLOPS_GRID)
    if case["kind"] != "batch":
        b += px * 4
    if case["kind"] == "adjoint":
        n = case["window"] or case["iters"]
        b += 2 * values * size + px * 2 * 8
        fl += px * min(n, case["iters"]) * FLOPS_BACK
    if case.get("kf_interval"):
        b += px * (16 + STATE_VALUES * size)
    return {"bytes": float(b), "flops": float(fl)}


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ---------------------------------------------------------------------------
# Planes come first ([6, H, W] vectors, [6, 6, H, W] matrices). One sweep (Eqs. 2-6): every factor is linearised at
# the current means, pairwise messages are damped, beliefs solved, means moved and message vectors transported.
def _mm(a, b):
    return (a.unsqueeze(2) * b.unsqueeze(0)).sum(1)


def _mv(a, x):
    return (a * x.unsqueeze(0)).sum(1)


def _tr(a):
    return a.transpose(0, 1)


def _inv_spd(a):
    """Inverse of symmetric positive definite [n, n, ...] by Gauss-Jordan elimination."""
    n = a.shape[0]
    eye = torch.eye(n, dtype=a.dtype, device=a.device).reshape((n, n) + (1,) * (a.dim() - 2)).expand_as(a)
    left, right = a, eye
    for k in range(n):
        lr, rr = left[k] / left[k, k], right[k] / left[k, k]
        col = left[:, k].unsqueeze(1)
        left = left - col * lr.unsqueeze(0)
        right = right - col * rr.unsqueeze(0)
        pick = (torch.arange(n, device=a.device) == k).reshape((n, 1) + (1,) * (a.dim() - 2))
        left, right = torch.where(pick, lr.unsqueeze(0), left), torch.where(pick, rr.unsqueeze(0), right)
    return right


def _hat(w):
    o = torch.zeros_like(w[0])
    return torch.stack([torch.stack([o, -w[2], w[1]]), torch.stack([w[2], o, -w[0]]), torch.stack([-w[1], w[0], o])])


def _series(t2, first):
    """sum_k (-t2)^k / (2k + first)!, for angles below about two radians."""
    out, c = torch.zeros_like(t2), 1.0 / math.factorial(first)
    for k in range(14):
        out = out + c * (-t2) ** k if k else out + c
        c /= (2 * k + first + 1) * (2 * k + first + 2)
    return out


def _eye3(w):
    return torch.eye(3, dtype=w.dtype, device=w.device).reshape((3, 3) + (1,) * (w.dim() - 1))


def _exp(xi):
    t2 = (xi[:3] ** 2).sum(0)
    k = _hat(xi[:3])
    k2 = _mm(k, k)
    A, B, C = _series(t2, 1), _series(t2, 2), _series(t2, 3)
    return _eye3(xi) + A * k + B * k2, _mv(_eye3(xi) + B * k + C * k2, xi[3:])


def _log(R, t):
    """Logarithm for rotations below half a turn: the angle over its sine by its power series below 0.3."""
    w = 0.5 * torch.stack([R[2, 1] - R[1, 2], R[0, 2] - R[2, 0], R[1, 0] - R[0, 1]])
    s2, c = (w * w).sum(0), 0.5 * (R[0, 0] + R[1, 1] + R[2, 2] - 1)
    small = (s2 < 0.09) & (c > 0)
    ratio, coef = torch.zeros_like(s2), 1.0
    sx = torch.where(small, s2, torch.zeros_like(s2))
    for k in range(22):  # asin(s)/s = sum_k (2k)! / (4^k k!^2 (2k + 1)) s^(2k)
        ratio = ratio + coef / (2 * k + 1) * (sx ** k if k else 1.0)
        coef *= (2 * k + 1) / (2.0 * k + 2)
    sl = torch.sqrt(torch.where(small, torch.ones_like(s2), s2))
    ratio = torch.where(small, ratio, torch.atan2(sl, torch.where(small, torch.ones_like(c), c)) / sl)
    th = w * ratio
    t2 = (th * th).sum(0)
    B = _series(t2, 2)
    # V^-1 = I - K/2 + D K^2 with D = (1 - A / (2 B)) / t^2, as a ratio of series: 2 B - A = t^2 E
    E = torch.zeros_like(t2)
    for k in range(13):
        c = 1.0 / math.factorial(2 * k + 3) - 2.0 / math.factorial(2 * k + 4)
        E = E + c * ((-t2) ** k if k else 1.0)
    D = E / (2 * B)
    K = _hat(th)
    return torch.cat([th, _mv(_eye3(th) - 0.5 * K + D * _mm(K, K), t)])


def _between(xj, R, t):
    """Log(Exp(xj)^-1 (R, t))."""
    Rj, tj = _exp(xj)
    return _log(_mm(_tr(Rj), R), _mv(_tr(Rj), t - tj))


def _shift(a, k, fill=0.0):
    """Values of the neighbour in direction k (left, right, up, down)."""
    out = torch.full_like(a, fill)
    if k == 0:
        return torch.cat([out[..., :1], a[..., :-1]], -1)
    if k == 1:
        return torch.cat([a[..., 1:], out[..., :1]], -1)
    if k == 2:
        return torch.cat([out[..., :1, :], a[..., :-1, :]], -2)
    return torch.cat([a[..., 1:, :], out[..., :1, :]], -2)


def _message(V, eta_v, r, lam):
    """A damping-free identity message: information lam (V + lam I)^-1 V and lam (V + lam I)^-1 (eta_v - V r)."""
    eye = torch.eye(6, dtype=V.dtype, device=V.device).reshape((6, 6) + (1,) * (V.dim() - 2))
    Ci = _inv_spd(V + lam * eye)
    L = lam * _mm(Ci, V)
    return 0.5 * (L + _tr(L)), lam * _mv(Ci, eta_v - _mv(V, r))


class _Exact:
    """The tracker in 64 bits, on images of shape [H, W]."""

    def __init__(self, case, w, h, dev):
        s = _strengths(case)
        # the library takes its strengths as float32
        f32 = lambda x: float(np.float32(x))  # noqa: E731
        self.lam = {k: 1.0 / f32(s["sigma_" + k]) ** 2 for k in "DPRNZ"}
        self.inv_sigma_D = 1.0 / f32(s["sigma_D"])
        self.K = [f32(c) for c in _camera(w, h)[:4]]
        self.w, self.h, self.tree, self.dev = w, h, _tree(case), dev
        self.u, self.v = _pixel_grid(w, h, dev)
        self.d_prior = 0.0
        self.levels = []
        if self.tree:
            while h > 1 or w > 1:
                h, w = (h + 1) // 2, (w + 1) // 2
                self.levels.append((h, w))

    def _zeros(self, *shape):
        return torch.zeros(*shape, dtype=torch.float64, device=self.dev)

    def keyframe(self, key, normals):
        h, w = self.h, self.w
        fx, fy, cx, cy = self.K
        self.I_s, n = key.double(), normals.double()
        nr = n[..., 0] * (self.u - cx) / fx + n[..., 1] * (self.v - cy) / fy + n[..., 2]
        ok = nr.abs() >= 1e-3
        ax = torch.where(ok, n[..., 0] / (fx * nr), torch.zeros_like(nr))
        ay = torch.where(ok, n[..., 1] / (fy * nr), torch.zeros_like(nr))
        self.m_x, self.m_y = self._zeros(h, w), self._zeros(h, w)
        self.m_x[:, :-1] = 0.5 * (ax[:, :-1] + ax[:, 1:])
        self.m_y[:-1] = 0.5 * (ay[:-1] + ay[1:])
        eye = torch.eye(6, dtype=torch.float64, device=self.dev)
        self.xi, self.d = self._zeros(6, h, w), self._zeros(h, w) + self.d_prior
        self.P = (self.lam["P"] * eye).reshape(6, 6, 1, 1).expand(6, 6, h, w)
        self.s = self._zeros(h, w) + self.lam["Z"]
        n_id = 1 if self.tree else 4
        self.L, self.e = [self._zeros(6, 6, h, w)] * n_id, [self._zeros(6, h, w)] * n_id
        self.nl, self.ne = [self._zeros(h, w)] * 4, [self._zeros(h, w)] * 4
        self.nodes = []
        for lvl, (hh, ww) in enumerate(self.levels, 1):
            self.nodes.append({"xi": self._zeros(6, hh, ww),
                               "P": (self.lam["P"] * 4.0 ** lvl * eye).reshape(6, 6, 1, 1).expand(6, 6, hh, ww),
                               "L": [self._zeros(6, 6, hh, ww)] * 5, "e": [self._zeros(6, hh, ww)] * 5})

    def _damp(self, new, old):
        return (1 - DAMPING) * new + DAMPING * old

    def _move(self, xi, R, t, tau):
        Rt, tt = _exp(tau)
        return _log(_mm(R, Rt), _mv(R, tt) + t)

    def _sweep(self, I_t, lam_D, lam_N):
        fx, fy, cx, cy = self.K
        h, w = self.h, self.w
        lam = self.lam
        R, t = _exp(self.xi)
        eye = torch.eye(6, dtype=torch.float64, device=self.dev).reshape(6, 6, 1, 1)
        M = (lam["P"] * eye).expand(6, 6, h, w)
        eb, ed = -lam["P"] * self.xi, -lam["Z"] * (self.d - self.d_prior)
        md = self._zeros(h, w) + lam["Z"]
        L, e, nl, ne = [], [], [], []
        inside = [_shift(torch.ones_like(self.d), k) for k in range(4)]
        if self.tree:
            par = self.nodes[0]
            up = lambda a: a.repeat_interleave(2, -2).repeat_interleave(2, -1)[..., :h, :w]  # noqa: E731
            sel = self._child_slot(h, w)
            mine = lambda lst: sum(up(x) * (sel == k) for k, x in enumerate(lst[:4]))  # noqa: E731
            r = _between(up(par["xi"]), R, t)
            Ln, en = _message(up(par["P"]) - mine(par["L"]), -mine(par["e"]), r, lam["R"])
            L.append(self._damp(Ln, self.L[0]))
            e.append(self._damp(en, self.e[0]))
        else:
            for k in range(4):
                r = _between(_shift(self.xi, k), R, t)
                Ln, en = _message(_shift(self.P - self.L[k ^ 1], k), -_shift(self.e[k ^ 1], k), r, lam["R"])
                L.append(self._damp(Ln, self.L[k]) * inside[k])
                e.append(self._damp(en, self.e[k]) * inside[k])
        for Lk, ek in zip(L, e):
            M, eb = M + Lk, eb + ek
        for k in range(4):
            sv, ev = _shift(self.s - self.nl[k ^ 1], k, 1.0), -_shift(self.ne[k ^ 1], k)
            m = (_shift(self.m_x, 0), self.m_x, _shift(self.m_y, 2), self.m_y)[k]
            rn = self.d - _shift(self.d, k) + (m if k in (0, 2) else -m)
            den = lam_N / (lam_N + sv)
            nl.append(self._damp(den * sv, self.nl[k]) * inside[k])
            ne.append(self._damp(den * (ev - sv * rn), self.ne[k]) * inside[k])
            md, ed = md + nl[k], ed + ne[k]
        # photometric factor
        z = torch.exp(self.d)
        Xs = torch.stack([z * (self.u - cx) / fx, z * (self.v - cy) / fy, z])
        Xt = _mv(R, Xs) + t
        iz = 1.0 / Xt[2]
        x, y = fx * Xt[0] * iz + cx, fy * Xt[1] * iz + cy
        valid = (Xt[2] > 1e-6) & (x >= -1e-3) & (x <= w - 1 + 1e-3) & (y >= -1e-3) & (y <= h - 1 + 1e-3)
        x, y = x.clamp(0, w - 1), y.clamp(0, h - 1)
        x0, y0 = x.detach().floor().long().clamp(0, w - 1), y.detach().floor().long().clamp(0, h - 1)
        x1, y1 = (x0 + 1).clamp(max=w - 1), (y0 + 1).clamp(max=h - 1)
        ax, ay = x - x0, y - y0

        def sample(img):
            return ((1 - ay) * ((1 - ax) * img[y0, x0] + ax * img[y0, x1]) +
                    ay * ((1 - ax) * img[y1, x0] + ax * img[y1, x1]))

        rep = torch.nn.functional.pad(I_t[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
        gx = sample(0.5 * (rep[1:-1, 2:] - rep[1:-1, :-2]))
        gy = sample(0.5 * (rep[2:, 1:-1] - rep[:-2, 1:-1]))
        res = self.I_s - sample(I_t)
        a = torch.stack([-gx * fx * iz, -gy * fy * iz, (gx * fx * Xt[0] + gy * fy * Xt[1]) * iz * iz])
        b = _mv(_tr(R), a)
        Jp = torch.cat([torch.stack([Xs[1] * b[2] - Xs[2] * b[1], Xs[2] * b[0] - Xs[0] * b[2],
                                     Xs[0] * b[1] - Xs[1] * b[0]]), b])
        Jd = (b * Xs).sum(0)
        mah = res.abs() * self.inv_sigma_D
        hub = mah > T_HUBER
        safe = torch.where(hub, mah, torch.ones_like(mah))
        wgt = torch.where(hub, (2 * T_HUBER * safe - T_HUBER ** 2) / (safe * safe), torch.ones_like(mah))
        alpha = torch.where(valid, wgt, torch.zeros_like(wgt)) * lam_D
        # belief: blockdiag(M, md) + alpha J J^T
        Mi = _inv_spd(M)
        hp, zp, hd, zd = _mv(Mi, eb), _mv(Mi, Jp), ed / md, Jd / md
        q = (Jp * zp).sum(0)
        coef = alpha * (res + (Jp * hp).sum(0) + Jd * hd) / (1 + alpha * (q + Jd * zd))
        tau, tau_d = hp - coef * zp, hd - coef * zd
        self.xi, self.d = self._move(self.xi, R, t, tau), self.d + tau_d
        self.P = M + (alpha * md / (md + alpha * Jd * Jd)) * (Jp.unsqueeze(1) * Jp.unsqueeze(0))
        self.s = md + alpha * Jd * Jd / (1 + alpha * q)
        old_L, old_e = self.L, self.e
        self.L, self.e = L, [ek - _mv(Lk, tau) for Lk, ek in zip(L, e)]
        self.nl, self.ne = nl, [b_ - a_ * tau_d for a_, b_ in zip(nl, ne)]
        return old_L, old_e

    def _child_slot(self, h, w):
        return 2 * (torch.arange(h, device=self.dev)[:, None] % 2) + torch.arange(w, device=self.dev)[None, :] % 2

    def _node_sweep(self, leaf):
        """Every node of every level from the state before the sweep; `leaf`: the pixels' state then."""
        eye = torch.eye(6, dtype=torch.float64, device=self.dev).reshape(6, 6, 1, 1)
        below, done = leaf, []
        for lvl, nd in enumerate(self.nodes, 1):
            hh, ww = nd["xi"].shape[1:]
            R, t = _exp(nd["xi"])
            L, e = [], []
            for k in range(4):  # from the children
                sub = lambda a: a[..., k // 2::2, k % 2::2]  # noqa: E731
                ch, cw = sub(below["xi"]).shape[1:]
                Ln, en = _message(sub(below["P"] - below["Lp"]), -sub(below["ep"]),
                                  _between(sub(below["xi"]), R[..., :ch, :cw], t[..., :ch, :cw]),
                                  self.lam["R"] * 4.0 ** (lvl - 1))
                pad = (0, ww - cw, 0, hh - ch)
                L.append(torch.nn.functional.pad(self._damp(Ln, nd["L"][k][..., :ch, :cw]), pad))
                e.append(torch.nn.functional.pad(self._damp(en, nd["e"][k][..., :ch, :cw]), pad))
            if lvl < len(self.nodes):  # from the parent
                up_nd = self.nodes[lvl]
                up = lambda a: a.repeat_interleave(2, -2).repeat_interleave(2, -1)[..., :hh, :ww]  # noqa: E731
                sel = self._child_slot(hh, ww)
                mine = lambda lst: sum(up(x) * (sel == k) for k, x in enumerate(lst[:4]))  # noqa: E731
                Ln, en = _message(up(up_nd["P"]) - mine(up_nd["L"]), -mine(up_nd["e"]),
                                  _between(up(up_nd["xi"]), R, t), self.lam["R"] * 4.0 ** lvl)
                L.append(self._damp(Ln, nd["L"][4]))
                e.append(self._damp(en, nd["e"][4]))
            else:
                L.append(nd["L"][4])
                e.append(nd["e"][4])
            lamP = self.lam["P"] * 4.0 ** lvl
            P = lamP * eye + sum(L)
            tau = _mv(_inv_spd(P), -lamP * nd["xi"] + sum(e))
            done.append({"xi": self._move(nd["xi"], R, t, tau), "P": P, "L": L,
                         "e": [ek - _mv(Lk, tau) for Lk, ek in zip(L, e)]})
            below = {"xi": nd["xi"], "P": nd["P"], "Lp": nd["L"][4], "ep": nd["e"][4]}
        return done

    def track(self, target, iters, lam_D=None, lam_N=None, detach_before=0, normals=None):
        I_t = target.double() if target.dtype != torch.float64 else target
        lam_D = self.lam["D"] if lam_D is None else lam_D
        lam_N = self.lam["N"] if lam_N is None else lam_N
        for i in range(iters):
            if i == detach_before:  # the state before is a constant
                for name in ("xi", "d", "P", "s"):
                    setattr(self, name, getattr(self, name).detach())
                for name in ("L", "e", "nl", "ne"):
                    setattr(self, name, [x.detach() for x in getattr(self, name)])
            with torch.set_grad_enabled(torch.is_grad_enabled() and i >= detach_before):
                xi, P = self.xi, self.P
                old_L, old_e = self._sweep(I_t, lam_D, lam_N)
                if self.tree:
                    self.nodes = self._node_sweep({"xi": xi, "P": P, "Lp": old_L[0], "ep": old_e[0]})
        pose = self.xi.mean((1, 2))
        if normals is not None:
            self.d_prior = float(self.d.mean())
            self.keyframe(target, normals)
        return pose, torch.exp(-self.d)


def exact(case, seed):
    """The first pass on a new state in 64 bits; None where it would need too long or too much memory."""
    dev = torch.device("cuda")
    n = case["iters"]
    if case["kind"] == "batch":
        poses = []
        for i, (w, h) in enumerate(_mix(case)):
            key, targets, normals, _ = _scene(w, h, seed * 1009 + i, NOISE, 2, dev)
            ref = _Exact(case, w, h, dev)
            ref.keyframe(key, normals)
            ref.track(targets[0], FIRST_SWEEPS)
            poses.append(ref.track(targets[1], n)[0])
        return {"poses": torch.stack(poses)}
    w, h = case["width"], case["height"]
    ref = _Exact(case, w, h, dev)
    if case["kind"] == "track":
        key, targets, normals, _ = _scene(w, h, seed, NOISE, 2, dev)
        ref.keyframe(key, normals)
        for target, sweeps in zip(targets, (FIRST_SWEEPS, n)):
            xi, inv = ref.track(target, sweeps, normals=normals if case["kf_interval"] else None)
        return {"xi": xi, "inv_depth": inv}
    window = min(case["window"] or n, n)
    if w * h * window > 160 * 120 * 30:  # the recorded sweeps would not fit
        return None
    key, targets, normals, inv_true = _scene(w, h, seed, NOISE_ADJOINT, 2, dev)
    with torch.no_grad():
        ref.keyframe(key, normals)
        ref.track(targets[0], FIRST_SWEEPS)
    I_s, I_t = key.double().requires_grad_(True), targets[1].double().requires_grad_(True)
    sig = [torch.tensor(float(np.float32(_strengths(case)[s])), dtype=torch.float64, device=dev, requires_grad=True)
           for s in ("sigma_D", "sigma_N")]
    ref.I_s = I_s
    xi, inv = ref.track(I_t, n, sig[0] ** -2, sig[1] ** -2, detach_before=n - window)
    g = torch.autograd.grad(_loss(xi, inv, inv_true), [I_s, I_t] + sig)
    return {"xi": xi.detach(), "inv_depth": inv.detach(), "d_key": g[0], "d_frame": g[1], "d_sigma_D": g[2],
            "d_sigma_N": g[3]}
