"""The work a user of this package has it do, as measurable cases.

``listed()`` names the standing cases, ``draw(rng)`` gives more of the same ranges.  ``prepare(case, seed)`` makes
what a program holds before the call (scans, keyframes, a tracker, a network), ``run(state)`` is one pass through
the public entry points, ``exact(case, seed)`` the same results in 64 bits from plain torch, and ``work(case)`` the
bytes and operations that a pass cannot do without.

All geometry is synthetic and seeded: a closed hall with pillars and crates, seen by a spinning lidar.  Keyframes
are rendered from the same hall (depth along pixel-centre rays, analytic normals, both with noise, sample counts
1 to 10, part of the sensor's field of view filled), so neither side of a comparison makes the other's inputs.
Decisions (pixel bins, neighbour tests, gates) are taken in FP32 by the package; ``exact`` takes the bins and
neighbour tests with the same published FP32 rule, one rounded operation at a time, and everything else in 64 bits.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2101_00585_gb300 as up
from paper_2101_00585_gb300 import proposal

DEV = "cuda"
F64 = torch.float64

# vertical half field of view of the sensors with few, 64 and many beams (degrees), as in the sweeps of 16, 64
# and 128 rows; keyframes span 45 degrees either way
SENSOR_FOV = ((16, 15.0), (64, 16.6), (1 << 30, 22.5))
KF_HALF_FOV = 45.0
KF_SHAPES = ((256, 1024), (512, 2048), (1024, 4096))  # a batch's keyframes, dealt in turn


def listed():
    return [
        # a small robot's 16-beam lidar in a room: the smallest sweep, latency of the registration loop
        dict(name="track_room", kind="track", rows=16, cols=512, kf_rows=256, kf_cols=512, f16=False, levels=0),
        # the ordinary stream: 64-beam sweeps against a 512 x 2048 keyframe, one call per sweep
        dict(name="track_tunnel", kind="track", rows=64, cols=1024, kf_rows=512, kf_cols=2048, f16=False, levels=0),
        # the largest stream: 128-beam sweeps, 4 M pixel keyframe held in 16-bit normals and counts
        dict(name="track_campus", kind="track", rows=128, cols=2048, kf_rows=1024, kf_cols=4096, f16=True, levels=0),
        # a sensor of odd size, normals smoothed by three a-trous levels before the registration
        dict(name="track_smoothed", kind="track", rows=43, cols=901, kf_rows=333, kf_cols=1777, f16=False, levels=3),
        # one registration from a rough guess, absolute error (IRLS): a loop closure's refinement
        dict(name="register_l1", kind="register", rows=64, cols=1024, kf_rows=512, kf_cols=2048, f16=False, l1=True),
        # many keyframes and hypotheses at once: relocalisation
        dict(name="batch_relocalise", kind="batch", rows=64, cols=1024, n_kf=12, n_hyp=8, f16=False),
        # the loop-closure grid search: 9 x 9 x 9 candidates on every fourth pixel
        dict(name="grid_search", kind="grid", rows=64, cols=1024, kf_rows=512, kf_cols=2048, n=729, stride=4,
             f16=False),
        # the keyframe update as a call of its own (mapping with poses from elsewhere)
        dict(name="fuse_update", kind="fuse", rows=64, cols=1024, kf_rows=512, kf_cols=2048, f16=False),
        # the check between two keyframes when the tracker switches
        dict(name="consistency", kind="consistency", kf_rows=512, kf_cols=2048, f16=False),
        # the learned start of one registration: a single pair, all latency
        dict(name="propose_one", kind="propose", batch=1),
        # proposals for a whole map's pairs
        dict(name="propose_many", kind="propose", batch=256),
        # one training step of the proposal network, as its training loop takes it
        dict(name="train_step", kind="train", batch=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["track", "track", "track", "register", "batch", "grid", "fuse", "consistency", "propose",
                       "train"])
    rows, cols = _log(rng, 16, 128), _log(rng, 512, 2048)
    kf_rows, kf_cols = _log(rng, 128, 1024), _log(rng, 512, 4096)
    f16 = rng.random() < 0.4
    kf = dict(kf_rows=kf_rows, kf_cols=kf_cols, f16=f16)
    if kind == "track":
        return dict(kind=kind, rows=rows, cols=cols, **kf, levels=rng.choice([0, 0, 1, 2, 3]))
    if kind == "register":
        return dict(kind=kind, rows=rows, cols=cols, **kf, l1=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind=kind, rows=min(rows, 64), cols=min(cols, 1024), n_kf=rng.randint(1, 12),
                    n_hyp=rng.randint(1, 8), f16=f16)
    if kind == "grid":
        return dict(kind=kind, rows=min(rows, 64), cols=min(cols, 1024), kf_rows=min(kf_rows, 512),
                    kf_cols=min(kf_cols, 2048), f16=f16, n=_log(rng, 20, 729), stride=rng.randint(4, 8))
    if kind == "fuse":
        return dict(kind=kind, rows=rows, cols=cols, **kf)
    if kind == "consistency":
        return dict(kind=kind, **kf)
    return dict(kind=kind, batch=_log(rng, 1, 256) if kind == "propose" else _log(rng, 8, 256))


# ----------------------------------------------------------------------------- geometry and the hall

def _pano(rows, cols, half_deg, r_min, r_max):
    h = math.radians(half_deg)
    return SimpleNamespace(rows=rows, cols=cols, el_top=np.float32(h), s_az=np.float32(cols / (2 * math.pi)),
                           s_el=np.float32(rows / (2 * h)), r_min=np.float32(r_min), r_max=np.float32(r_max))


def _sensor(rows, cols):
    half = next(f for n, f in SENSOR_FOV if rows <= n)
    return _pano(rows, cols, half, 0.3, 120.0)


def _keyframe(rows, cols):
    return _pano(rows, cols, KF_HALF_FOV, 0.3, 150.0)


def _dirs(p):
    """FP64 unit rays of a panorama's pixel centres [rows, cols, 3]."""
    el = float(p.el_top) - (torch.arange(p.rows, device=DEV, dtype=F64) + 0.5) / float(p.s_el)
    az = math.pi - (torch.arange(p.cols, device=DEV, dtype=F64) + 0.5) / float(p.s_az)
    ce, se = torch.cos(el)[:, None], torch.sin(el)[:, None]
    return torch.stack([ce * torch.cos(az), ce * torch.sin(az), se.expand(p.rows, p.cols)], -1)


def _pose(yaw, pitch, roll, t):
    cy, sy, cp, sp, cr, sr = (f(a) for a in (yaw, pitch, roll) for f in (math.cos, math.sin))
    R = (np.array([[cy, -sy, 0], [sy, cy, 0], [0, 0, 1]]) @ np.array([[cp, 0, sp], [0, 1, 0], [-sp, 0, cp]])
         @ np.array([[1, 0, 0], [0, cr, -sr], [0, sr, cr]]))
    return np.hstack([R, np.asarray(t, float)[:, None]])


def _mul(A, B):
    return np.hstack([A[:, :3] @ B[:, :3], A[:, :3] @ B[:, 3:] + A[:, 3:]])


def _inv(A):
    return np.hstack([A[:, :3].T, -A[:, :3].T @ A[:, 3:]])


class _Hall:
    """A closed hall with pillars along both sides and crates on the floor; ray casting in FP64."""

    def __init__(self, rng):
        self.half = np.array([rng.uniform(22, 30), rng.uniform(4.5, 7.0), 0.0])
        self.top = rng.uniform(3.5, 5.0)
        side = rng.choice([-1.0, 1.0], 14)
        self.pillars = [(x, s * rng.uniform(0.55, 0.9) * self.half[1], rng.uniform(0.15, 0.45))
                        for x, s in zip(np.linspace(-20, 20, 14) + rng.uniform(-1, 1, 14), side)]
        self.crates = []
        for s in rng.choice([-1.0, 1.0], 8):
            c = np.array([rng.uniform(-18, 18), s * rng.uniform(2.6, 4.0), 0.0])
            h = np.array([rng.uniform(0.3, 1.0), rng.uniform(0.3, 0.8), rng.uniform(0.4, 1.6)])
            self.crates.append((c - h, c + h))

    def cast(self, P, dirs):
        """Range and world normal of the first surface along sensor-frame rays ``dirs`` from pose P."""
        R = torch.as_tensor(P[:, :3], device=DEV)
        o = [float(v) for v in P[:, 3]]
        d = dirs @ R.T
        best = torch.full(d.shape[:-1], 1e9, dtype=F64, device=DEV)
        nrm = torch.zeros_like(d)

        def take(t, hit, n):
            m = hit & (t > 1e-4) & (t < best)
            best[m] = t[m]
            nrm[m] = (n[m] if isinstance(n, torch.Tensor) else torch.tensor(n, dtype=F64, device=DEV))

        lo, hi = (-self.half[0], -self.half[1], 0.0), (self.half[0], self.half[1], self.top)
        for k in range(3):
            for plane, s in ((lo[k], 1.0), (hi[k], -1.0)):
                n = [0.0, 0.0, 0.0]
                n[k] = s
                take((plane - o[k]) / d[..., k], d[..., k] * s < 0, n)
        for x, y, r in self.pillars:
            fx, fy = o[0] - x, o[1] - y
            a = d[..., 0] ** 2 + d[..., 1] ** 2
            b = fx * d[..., 0] + fy * d[..., 1]
            disc = b * b - a * (fx * fx + fy * fy - r * r)
            t = (-b - disc.clamp_min(0).sqrt()) / a
            n = torch.stack([(fx + t * d[..., 0]) / r, (fy + t * d[..., 1]) / r, torch.zeros_like(t)], -1)
            take(t, disc > 0, n)
        for a, b in self.crates:
            t0 = torch.stack([(torch.where(d[..., k] > 0, a[k], b[k]) - o[k]) / d[..., k] for k in range(3)], -1)
            t1 = torch.stack([(torch.where(d[..., k] > 0, b[k], a[k]) - o[k]) / d[..., k] for k in range(3)], -1)
            t, axis = t0.max(-1)
            n = torch.zeros_like(d).scatter_(-1, axis[..., None], -torch.sign(d.gather(-1, axis[..., None])))
            take(t, t < t1.min(-1).values, n)
        return best, nrm @ R  # the normal in the sensor frame


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFFFFFF)


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=F64)


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV, dtype=F64)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _scan(hall, P, p, g):
    """FP32 points (x, y, z, valid) in the order a spinning sensor emits them: 2 cm noise, 2 % lost returns."""
    dirs = _dirs(p).transpose(0, 1).reshape(-1, 3)
    t, _ = hall.cast(P, dirs)
    t = t + 0.02 * _randn(g, t.numel())
    ok = (_rand(g, t.numel()) >= 0.02) & (t > float(p.r_min)) & (t < float(p.r_max))
    pts = torch.cat([dirs * t[:, None], torch.ones_like(t)[:, None]], 1) * ok[:, None]
    return pts.float().contiguous()


def _sweep_image(hall, P, p, g, f16):
    """A sweep as the package holds it: pixel points [rows, cols, 4] and normals."""
    dirs = _dirs(p)
    t, n = hall.cast(P, dirs)
    t = t + 0.02 * _randn(g, p.rows, p.cols)
    n = _unit(n + 0.04 * _randn(g, p.rows, p.cols, 3))
    ok = (_rand(g, p.rows, p.cols) >= 0.02)[..., None]
    one = torch.ones_like(t)[..., None]
    pix = (torch.cat([dirs * t[..., None], one], -1) * ok).float()
    nrm = (torch.cat([n, one], -1) * ok).float()
    return pix.contiguous(), (nrm.half() if f16 else nrm).contiguous()


def _kf_image(hall, P, p, g, f16, sensor_half, fill=0.6):
    """A keyframe some sweeps old: ``fill`` of the sensor's field of view holds samples, counted 1 to 10."""
    t, n = hall.cast(P, _dirs(p))
    t = t + 0.01 * _randn(g, p.rows, p.cols)
    n = _unit(n + 0.04 * _randn(g, p.rows, p.cols, 3))
    el = float(p.el_top) - (torch.arange(p.rows, device=DEV, dtype=F64) + 0.5) / float(p.s_el)
    seen = (el.abs() < math.radians(sensor_half + 2.0))[:, None] & (_rand(g, p.rows, p.cols) < fill)
    w = torch.randint(1, 11, (p.rows, p.cols), generator=g, device=DEV).to(F64)
    depth = torch.where(seen, t, torch.zeros_like(t)).float()
    nw = (torch.cat([n, w[..., None]], -1) * seen[..., None]).float()
    return depth.contiguous(), (nw.half() if f16 else nw).contiguous()


def _dev_pose(T):
    return torch.tensor(np.asarray(T).reshape(12), dtype=F64, device=DEV)


TRACK_SCANS = 6  # a stream's scans, driven forth and back


def _world(case, seed):
    """Everything random of a case, from the seed alone."""
    rng = np.random.default_rng(int(seed) & 0x7FFFFFFFFFFF)
    g = _gen(seed)
    hall = _Hall(rng)
    w = SimpleNamespace(rng=rng, g=g, hall=hall, f16=bool(case.get("f16")))
    P_kf = _pose(rng.uniform(-0.2, 0.2), 0.01, -0.01, [rng.uniform(-4, 4), rng.uniform(-0.5, 0.5), 1.5])
    if "rows" in case:
        w.sp = _sensor(case["rows"], case["cols"])
    if "kf_rows" in case:
        w.kp = _keyframe(case["kf_rows"], case["kf_cols"])
        half = math.degrees(float(w.sp.el_top)) if "rows" in case else 16.6
        w.depth, w.nw = _kf_image(hall, P_kf, w.kp, g, w.f16, half)
    kind = case["kind"]
    if kind == "track":
        # 10 cm and half a degree from sweep to sweep; the tracker has already followed the sweeps before
        step = _pose(math.radians(0.5), 0.0, 0.0, [0.1, 0.004, 0.0])
        T = [_pose(0.03, 0.004, 0.0, [0.6, 0.05, 0.0])]
        for _ in range(TRACK_SCANS):
            T.append(_mul(T[-1], _mul(step, _pose(*(0.002 * rng.standard_normal(3)), 0.01 * rng.standard_normal(3)))))
        w.prev, w.motion = T[0], step
        w.scans = [_scan(hall, _mul(P_kf, t), w.sp, g) for t in T[1:]]
    elif kind in ("register", "grid", "fuse"):
        T = _pose(0.05, 0.01, -0.005, [0.7, -0.15, 0.02])
        w.pix, w.nrm = _sweep_image(hall, _mul(P_kf, T), w.sp, g, w.f16)
        w.T = T
        off = {"register": (0.02, 0.12), "grid": (0.05, 0.3), "fuse": (0.0002, 0.003)}[kind]
        w.T0 = _mul(T, _pose(off[0], 0.2 * off[0], 0.0, [off[1], -0.5 * off[1], 0.1 * off[1]]))
        if kind == "grid":
            w.xi = (torch.rand((case["n"], 6), generator=g, device=DEV) - 0.5) \
                * torch.tensor([0.04, 0.04, 0.3, 1.2, 1.2, 0.2], device=DEV)
    elif kind == "consistency":
        # the second keyframe 3 m on, in the same hall with some crates moved
        w.T = _pose(0.1, 0.0, 0.0, [3.0, 0.3, 0.0])
        hall.crates = [(a + [1.5, 0, 0], b + [1.5, 0, 0]) if i % 3 == 0 else (a, b)
                       for i, (a, b) in enumerate(hall.crates)]
        w.depth_b, w.nw_b = _kf_image(hall, _mul(P_kf, w.T), w.kp, g, w.f16, 16.6)
    elif kind == "batch":
        w.pix, w.nrm = _sweep_image(hall, P_kf, w.sp, g, w.f16)
        w.kfs, w.T0 = [], []
        half = math.degrees(float(w.sp.el_top))
        for i in range(case["n_kf"]):
            T = _pose(rng.uniform(-0.5, 0.5), 0.01, 0.0, [rng.uniform(-2, 2), rng.uniform(-0.5, 0.5), 0.0])
            kp = _keyframe(*KF_SHAPES[i % 3])
            w.kfs.append((kp, *_kf_image(hall, _mul(P_kf, _inv(T)), kp, g, w.f16, half)))
            for _ in range(case["n_hyp"]):
                w.T0.append(_mul(T, _pose(rng.uniform(-0.2, 0.2), 0.0, 0.0, rng.uniform(-1, 1, 3) * [0.8, 0.6, 0.1])))
    return w


def _net_inputs(case, seed):
    """Pairs of downsampled panoramas [B, 64, 256, 8] BF16, their poses, and a network some steps into training."""
    g = _gen(seed)
    B = case["batch"]
    ph = 6.28 * torch.rand((B, 2, 3, 1, 1), generator=g, device=DEV)
    v = torch.linspace(-1, 1, 64, device=DEV)[:, None]
    u = torch.linspace(0, 2 * math.pi, 257, device=DEV)[None, :256]
    f = (torch.sin(u + ph[:, :, 0]) + 0.5 * torch.sin(3 * u + ph[:, :, 1] + v) + 0.3 * torch.cos(2 * v + ph[:, :, 2]))
    depth = (0.5 + 0.2 * f) * (1 + 0.02 * torch.randn(f.shape, generator=g, device=DEV))
    n = torch.stack([torch.sin(u + f), torch.cos(u + f).expand_as(f), 0.4 * torch.sin(2 * f + v)], -1)
    n = n / n.norm(dim=-1, keepdim=True)
    x = torch.cat([depth[..., None], n], -1)  # [B, 2, 64, 256, 4]
    x = x * (torch.rand(f.shape, generator=g, device=DEV) < 0.9)[..., None]
    x = x.permute(0, 2, 3, 1, 4).reshape(B, 64, 256, 8).to(torch.bfloat16).contiguous()
    xi = (torch.rand((B, 6), generator=g, device=DEV) - 0.5) * torch.tensor([0.5] * 3 + [1.5] * 3, device=DEV)
    gc = torch.Generator().manual_seed(int(seed) & 0x7FFFFFFF)
    ch = proposal.CHANNELS
    parts = []
    for ci, co in zip(ch[:-1], ch[1:]):
        parts += [torch.randn(co * 9 * ci, generator=gc) * math.sqrt(2.0 / (9 * ci)),
                  0.05 * torch.randn(co, generator=gc)]
    parts += [0.02 * torch.randn(6 * 128, generator=gc), 0.01 * torch.randn(6, generator=gc)]
    params = torch.cat(parts).float()
    m = 0.01 * torch.randn(params.numel(), generator=gc)
    s = 0.02 + 0.05 * torch.rand(params.numel(), generator=gc)
    return x, xi.contiguous(), dict(params=params, m=m, v=s * s, step=400)


LR = 2e-4


def _params(case):
    """The registration settings of a case, as a program would pass them."""
    if case["kind"] == "batch":  # hypotheses far off: a wide gate for five steps, then the usual one
        return up.Params(d_max=1.0, coarse_iters=5, d_max_fine=0.5)
    if case["kind"] == "register":
        return up.Params(loss=1 if case["l1"] else 0)
    return up.Params(atrous_levels=int(case.get("levels", 0)))


# ----------------------------------------------------------------------------- the calls

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("propose", "train"):
        x, xi, sd = _net_inputs(case, seed)
        net = proposal.PoseNet(case["batch"], params=sd["params"])
        net.load_state_dict(sd)
        return SimpleNamespace(kind=kind, net=net, x=x, xi=xi)
    w = _world(case, seed)
    prec = up.F16 if w.f16 else up.F32
    prm = _params(case)
    s = SimpleNamespace(kind=kind, prm=prm)
    if kind == "track":
        s.trk = up.Tracker(w.sp, w.kp, prm, precision=prec)
        s.trk.kf.set(w.depth, w.nw)
        s.trk.prev.copy_(_dev_pose(w.prev))
        s.trk.motion.copy_(_dev_pose(w.motion))
        s.scans = w.scans + w.scans[-2:0:-1]
        s.at = 0
        return s
    if kind == "consistency":
        s.a, s.b = up.KeyframeBuffer(w.kp, precision=prec), up.KeyframeBuffer(w.kp, precision=prec)
        s.a.set(w.depth, w.nw)
        s.b.set(w.depth_b, w.nw_b)
        s.T = _dev_pose(w.T)
        return s
    s.sw = up.SweepFrame(w.sp, precision=prec)
    s.sw.set(w.pix, w.nrm)
    if kind == "batch":
        s.kfs = [up.KeyframeBuffer(kp, precision=prec) for kp, _, _ in w.kfs]
        for k, (_, d, nw) in zip(s.kfs, w.kfs):
            k.set(d, nw)
        s.batch = up.Batch(s.sw, s.kfs, case["n_hyp"])
        s.T0 = torch.tensor(np.stack(w.T0).reshape(-1, 12), dtype=F64, device=DEV)
        return s
    s.kf = up.KeyframeBuffer(w.kp, precision=prec)
    s.kf.set(w.depth, w.nw)
    s.T0 = _dev_pose(w.T0)
    if kind == "register":
        s.state = up.IcpState(s.kf)
    elif kind == "grid":
        s.xi, s.stride = w.xi.contiguous(), case["stride"]
    return s


def _record(stats):
    """A registration record's device values: A (21), b (6), sse; inliers and valid."""
    return stats[..., :224].view(F64), stats[..., 224:240].view(torch.int64)


def run(s):
    if s.kind == "track":
        s.trk.track(s.scans[s.at % len(s.scans)])
        s.at += 1
        t = s.trk
        sums, counts = _record(t.state.stats)
        return dict(pose=t.state.pose, motion=t.motion, prev=t.prev, sums=sums, counts=counts, kf_depth=t.kf.depth,
                    kf_nw=t.kf.nw, depth=t.sw.depth, idx=t.sw.idx, pix=t.sw.pix, nrm=t.sw.nrm)
    if s.kind == "register":
        s.state.pose.copy_(s.T0)
        up.icp(s.kf, s.sw, s.state, s.prm)
        sums, counts = _record(s.state.stats)
        return dict(pose=s.state.pose, sums=sums, counts=counts)
    if s.kind == "batch":
        s.batch.run(s.T0, s.prm)
        sums, counts = _record(s.batch.stats)
        return dict(poses=s.batch.poses, sums=sums, counts=counts)
    if s.kind == "grid":
        poses = up.grid_candidates(s.T0, s.xi)
        scores, best, best_pose = up.grid_score(s.kf, s.sw, poses, s.prm, s.stride)
        return dict(poses=poses, scores=scores, best=best, best_pose=best_pose)
    if s.kind == "fuse":
        up.fuse(s.kf, s.sw, s.T0, s.prm)
        return dict(depth=s.kf.depth, nw=s.kf.nw)
    if s.kind == "consistency":
        removed, fa, fb = up.keyframe_consistency(s.a, s.b, s.T)
        return dict(removed=removed, flags_a=fa, flags_b=fb, depth_a=s.a.depth, nw_a=s.a.nw, depth_b=s.b.depth,
                    nw_b=s.b.nw)
    if s.kind == "propose":
        out = s.net.forward(s.x)
        return dict(xi=out, poses=proposal.poses_from_twists(out))
    loss = s.net.train_step(s.x, s.xi, LR)
    n = s.net
    return dict(loss=loss, out=n.out, grads=n.grads, params=n.params, m=n.m, v=n.v)


# bytes of a pair's activations: input, the four layers' outputs
_ACT = [64 * 256 * 8 * 2] + [(64 >> l) * (256 >> l) * c * 2 for l, c in ((1, 32), (2, 64), (3, 128), (4, 128))]
_MACS = [(64 >> l) * (256 >> l) * 9 * ci * co for l, ci, co in ((1, 8, 32), (2, 32, 64), (3, 64, 128), (4, 128, 128))]
_N_PARAMS = sum(9 * ci * co + co for ci, co in ((8, 32), (32, 64), (64, 128), (128, 128))) + 6 * 128 + 6
# FP32 operations of one projective correspondence: transform, binning rule, gates, normal equations
_PAIR_FLOPS = 200


def work(case):
    kind = case["kind"]
    if kind in ("propose", "train"):
        B, macs = case["batch"], 2 * sum(_MACS)
        if kind == "propose":
            return dict(bytes=B * (_ACT[0] + 24 + 96) + 4 * _N_PARAMS, flops=B * macs)
        # forward, weight gradients, data gradients of all layers but the first; Adam reads and writes its state
        return dict(bytes=B * (_ACT[0] + 48) + 32 * _N_PARAMS, flops=B * (3 * macs - 2 * _MACS[0]))
    ns = case.get("rows", 0) * case.get("cols", 0)
    nb = 8 if case.get("f16") else 16
    sweep = ns * (16 + nb)
    if kind == "batch":
        shapes = [KF_SHAPES[i % 3] for i in range(case["n_kf"])]
        px = sum(r * c for r, c in shapes)
        samples = px * 0.25
        return dict(bytes=px * 4 + samples * nb + sweep + 96 * 2 * case["n_kf"] * case["n_hyp"],
                    flops=samples * case["n_hyp"] * 10 * _PAIR_FLOPS)
    px = case["kf_rows"] * case["kf_cols"]
    samples = px * 0.25  # about a quarter of a keyframe holds samples
    kf = px * 4 + samples * nb
    if kind == "track":
        return dict(bytes=ns * 16 + ns * (8 + 16 + nb) + 2 * kf, flops=samples * 8 * _PAIR_FLOPS)
    if kind == "register":
        return dict(bytes=kf + sweep, flops=samples * 10 * _PAIR_FLOPS)
    if kind == "fuse":
        return dict(bytes=2 * kf + sweep, flops=(samples + ns) * 120)
    if kind == "consistency":
        return dict(bytes=2 * (px * 5 + samples * 0.1 * (4 + nb)), flops=2 * samples * 100)
    n, st = case["n"], case["stride"]
    return dict(bytes=kf / st ** 2 + sweep + n * 200, flops=samples / st ** 2 * n * 120)


# ----------------------------------------------------------------------------- 64-bit results

def _atan2_rule(y, x):
    """The binning rule's FP32 atan2: octant reduction and a fixed polynomial, every operation rounded."""
    ax, ay = x.abs(), y.abs()
    swap = ay > ax
    mx, mn = torch.where(swap, ay, ax), torch.where(swap, ax, ay)
    t = torch.where(mx == 0, torch.zeros_like(mx), mn / mx)
    q = t * t
    p = torch.full_like(q, 0.0028662257)
    for c in (-0.0161657367, 0.0429096138, -0.0752896400, 0.1065626393, -0.1420889944, 0.1999355085, -0.3333314528,
              1.0):
        p = p * q
        p = p + torch.tensor(c, dtype=torch.float32, device=DEV)
    a = t * p
    a = torch.where(swap, torch.tensor(math.pi / 2, dtype=torch.float32, device=DEV) - a, a)
    a = torch.where(x < 0, torch.tensor(math.pi, dtype=torch.float32, device=DEV) - a, a)
    return torch.where(y < 0, -a, a)


def _bin(q, p):
    """Row, column, FP32 range and acceptance of FP32 points [..., 3] in panorama p."""
    x, y, z = q.unbind(-1)
    xy2 = x * x
    xy2 = xy2 + y * y
    r = (xy2 + z * z).sqrt()
    f32 = lambda v: torch.tensor(float(v), dtype=torch.float32, device=DEV)  # noqa: E731
    fc = (f32(math.pi) - _atan2_rule(y, x)) * f32(p.s_az)
    fr = (f32(p.el_top) - _atan2_rule(z, xy2.sqrt())) * f32(p.s_el)
    ok = (r >= f32(p.r_min)) & (r <= f32(p.r_max)) & (fr >= 0) & (fr < float(p.rows))
    row = torch.where(ok, fr, torch.zeros_like(fr)).floor().long()
    col = fc.floor().long()
    return row, torch.where(col >= p.cols, col - p.cols, col).clamp(0, p.cols - 1), r, ok


def _rot32(T, v, inverse=False):
    """T v (or T^-1 v) for FP32 points in the rule's order of rounded operations."""
    r = torch.as_tensor(np.asarray(T, np.float64), device=DEV).float()
    if inverse:
        d = v - r[:, 3]
        return torch.stack([(r[0, i] * d[..., 0] + r[1, i] * d[..., 1]) + r[2, i] * d[..., 2] for i in range(3)], -1)
    return torch.stack([((r[i, 0] * v[..., 0] + r[i, 1] * v[..., 1]) + r[i, 2] * v[..., 2]) + r[i, 3]
                        for i in range(3)], -1)


def _kf_points(depth, p):
    d = _dirs32(p)
    return depth[..., None] * d


def _dirs32(p):
    """Pixel rays from the FP32 table of row and column cosines and sines, products rounded."""
    el = float(p.el_top) - (torch.arange(p.rows, device=DEV, dtype=F64) + 0.5) / float(p.s_el)
    az = math.pi - (torch.arange(p.cols, device=DEV, dtype=F64) + 0.5) / float(p.s_az)
    ce, se, ca, sa = (f(a).float() for a in (el, az) for f in (torch.cos, torch.sin))
    return torch.stack([ce[:, None] * ca, ce[:, None] * sa, se[:, None].expand(p.rows, p.cols)], -1)


def _project64(pts, p):
    """Depth, winner index and point of every pixel of a scan."""
    row, col, r, ok = _bin(pts[:, :3], p)
    ok = ok & (pts[:, 3] != 0)
    key = (r.view(torch.int32).long() << 32) | torch.arange(pts.shape[0], device=DEV)
    none = torch.iinfo(torch.int64).max
    best = torch.full((p.rows * p.cols,), none, dtype=torch.int64, device=DEV)
    best.scatter_reduce_(0, (row * p.cols + col)[ok], key[ok], "amin")
    has = (best != none).view(p.rows, p.cols)
    idx = torch.where(has, (best & 0xFFFFFFFF).view(p.rows, p.cols), torch.full_like(has, -1, dtype=torch.int64))
    xyz = pts[idx.clamp_min(0), :3]
    depth32 = torch.where(has, (best >> 32).int().view(torch.float32).view(p.rows, p.cols), torch.zeros_like(r[0]))
    return depth32, idx, torch.where(has[..., None], xyz, torch.zeros_like(xyz)), has


def _normals64(depth, xyz, has, p, prm):
    d64 = xyz.double()
    lim = torch.tensor(prm.jump_rel, dtype=torch.float32, device=DEV) * depth
    lim = lim + torch.tensor(prm.jump_abs, dtype=torch.float32, device=DEV)

    def side(shift, axis):
        ok = torch.roll(has, shift, axis) & ~((torch.roll(depth, shift, axis) - depth).abs() > lim)
        if axis == 0:
            ok[-1 if shift < 0 else 0] = False
        return torch.roll(d64, shift, axis), ok

    (qr, okr), (ql, okl), (qd, okd), (qu, oku) = side(-1, 1), side(1, 1), side(-1, 0), side(1, 0)
    a = torch.where(okr[..., None], qr - d64, d64 - ql)
    b = torch.where(okd[..., None], qd - d64, d64 - qu)
    n = torch.linalg.cross(a, b)
    nn = n.norm(dim=-1)
    ok = has & (okr | okl) & (okd | oku) & (nn >= prm.min_cross * a.norm(dim=-1) * b.norm(dim=-1)) & (nn > 0)
    n = n / nn.clamp_min(1e-300)[..., None]
    n = torch.where(((n * d64).sum(-1) > 0)[..., None], -n, n)
    return torch.cat([n, torch.ones_like(nn)[..., None]], -1) * ok[..., None]


def _atrous64(xyz, nrm, prm):
    h = torch.tensor([1, 4, 6, 4, 1], dtype=F64, device=DEV) / 16
    P = xyz.double()
    sc = (prm.atrous_sigma_x ** 2) * (P * P).sum(-1).clamp_min(1e-300)
    for level in range(prm.atrous_levels):
        N, ok, acc = nrm[..., :3], nrm[..., 3] != 0, torch.zeros_like(nrm[..., :3])
        for dy in range(-2, 3):
            for dx in range(-2, 3):
                sh = (-dy << level, -dx << level)
                Nq, Pq, okq = (torch.roll(v, sh, (0, 1)) for v in (N, P, ok))
                okq = okq.clone()
                if sh[0]:
                    k = min(abs(sh[0]), okq.shape[0])
                    okq[-k:] &= sh[0] > 0
                    okq[:k] &= sh[0] < 0
                w = h[dy + 2] * h[dx + 2] * torch.exp(-((N - Nq) ** 2).sum(-1) / prm.atrous_sigma_n ** 2
                                                      - (N * (Pq - P)).sum(-1) ** 2 / sc)
                acc += torch.where(okq, w, torch.zeros_like(w))[..., None] * Nq
        n = acc / acc.norm(dim=-1, keepdim=True).clamp_min(1e-300)
        nrm = torch.cat([n, torch.ones_like(n[..., :1])], -1) * ok[..., None]
    return nrm


def _se3_exp(xi):
    w, v = xi[:3], xi[3:]
    W = np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])
    th = np.linalg.norm(w)
    if th < 1e-4:
        A, B, C = 1 - th ** 2 / 6, 0.5 - th ** 2 / 24, 1 / 6 - th ** 2 / 120
    else:
        A, B, C = math.sin(th) / th, (1 - math.cos(th)) / th ** 2, (th - math.sin(th)) / th ** 3
    return np.hstack([np.eye(3) + A * W + B * W @ W, ((np.eye(3) + B * W + C * W @ W) @ v)[:, None]])


def _pairs(T, s, pix, nrm, p):
    """The sweep sample that each keyframe point s (FP32) bins into: T s2, R m, and whether there is one."""
    row, col, _, ok = _bin(_rot32(T, s, inverse=True), p)
    P, m = pix[row, col], nrm[row, col]
    ok = ok & (P[..., 3] != 0) & (m[..., 3] != 0)
    T32 = torch.as_tensor(np.asarray(T, np.float64), device=DEV).float().double()
    return P[..., :3].double() @ T32[:, :3].T + T32[:, 3], m[..., :3].double() @ T32[:, :3].T, ok


def _icp64(kp, depth, nw, sp, pix, nrm, T, prm):
    """Point-to-plane registration: pose, [A, b, sse] of the last linearisation."""
    n = nw[..., :3].float()
    hold = (depth > 0) & (((n[..., 0] * n[..., 0] + n[..., 1] * n[..., 1]) + n[..., 2] * n[..., 2]) > 0.25)
    s, n = _kf_points(depth, kp)[hold], n[hold].double()
    iu = np.triu_indices(6)
    for _ in range(prm.max_iters):
        p, Rm, ok = _pairs(T, s, pix, nrm, sp)
        e = p - s.double()
        ok = ok & ((e * e).sum(-1) <= prm.d_max ** 2) & ((Rm * n).sum(-1) >= prm.cos_theta_max)
        r = (e * n).sum(-1)[ok]
        J = torch.cat([torch.linalg.cross(p[ok], n[ok]), n[ok]], -1)
        w = 1.0 / r.abs().clamp_min(prm.loss_delta) if prm.loss else torch.ones_like(r)
        A, b = (J.T @ (J * w[:, None])).cpu().numpy(), (J.T @ (w * r)).cpu().numpy()
        sums = np.concatenate([A[iu], b, [float((w * r * r).sum())]])
        xi = np.linalg.solve(A, -b)
        T = _mul(_se3_exp(xi), T)
        if np.linalg.norm(xi[:3]) < prm.eps_rot and np.linalg.norm(xi[3:]) < prm.eps_trans:
            break
    return T, torch.from_numpy(sums)


def _fuse64(kp, depth, nw, sp, pix, nrm, T, prm):
    """The keyframe after the sweep is averaged in and empty pixels are filled."""
    d, out = depth.double(), nw.double().clone()
    hold = (out[..., 3] > 0) & (depth > 0)
    s = _kf_points(depth, kp)
    p, Rm, ok = _pairs(T, s, pix, nrm, sp)
    e = p - s.double()
    ok = ok & hold & ((e * e).sum(-1) <= prm.fuse_d_max ** 2) & ((Rm * out[..., :3]).sum(-1) >= prm.fuse_cos_theta_max)
    w = out[..., 3]
    nd = torch.where(ok, (w * d + p.norm(dim=-1)) / (w + 1), d)
    nn = _unit(w[..., None] * out[..., :3] + Rm)
    out[ok] = torch.cat([nn, (w + 1).clamp_max(prm.w_max)[..., None]], -1)[ok]
    row, col, r, okf = _bin(_rot32(T, pix[..., :3].reshape(-1, 3)), kp)
    okf = okf & (pix[..., 3].reshape(-1) != 0) & (nrm[..., 3].reshape(-1) != 0)
    px = row * kp.cols + col
    okf = okf & (depth.reshape(-1)[px] == 0)
    key = (r.view(torch.int32).long() << 32) | torch.arange(r.numel(), device=DEV)
    none = torch.iinfo(torch.int64).max
    best = torch.full((kp.rows * kp.cols,), none, dtype=torch.int64, device=DEV)
    best.scatter_reduce_(0, px[okf], key[okf], "amin")
    at = (best != none).nonzero()[:, 0]
    j = best[at] & 0xFFFFFFFF
    T32 = torch.as_tensor(np.asarray(T, np.float64), device=DEV).float().double()
    xyz = pix[..., :3].reshape(-1, 3)[j].double() @ T32[:, :3].T + T32[:, 3]
    m = _unit(nrm[..., :3].reshape(-1, 3)[j].double() @ T32[:, :3].T)
    nd.view(-1)[at] = xyz.norm(dim=-1)
    out.view(-1, 4)[at] = torch.cat([m, torch.ones_like(m[:, :1])], -1)
    return nd, out


def _net64(x, params):
    """The network in 64 bits on plain convolutions; ``params`` flat, differentiable."""
    ch, o = proposal.CHANNELS, 0
    a = x.double().permute(0, 3, 1, 2)

    def take(*shape):
        nonlocal o
        n = math.prod(shape)
        o += n
        return params[o - n:o].view(*shape)

    for ci, co in zip(ch[:-1], ch[1:]):
        wt, b = take(co, 3, 3, ci).permute(0, 3, 1, 2), take(co)
        cols = torch.nn.functional.unfold(a, 3, padding=1, stride=2)
        y = wt.reshape(co, -1) @ cols
        a = torch.relu(y.view(a.shape[0], co, a.shape[2] // 2, a.shape[3] // 2) + b[:, None, None])
    wf, bf = take(6, 128), take(6)
    return a.mean((2, 3)) @ wf.T + bf


def _exact_net(case, seed):
    x, xi, sd = _net_inputs(case, seed)
    p = sd["params"].to(DEV).double().requires_grad_(case["kind"] == "train")
    parts = x.split(32)
    if case["kind"] == "propose":
        out = torch.cat([_net64(c, p) for c in parts])
        poses = np.stack([_se3_exp(v).reshape(12) for v in out.cpu().numpy()])
        return dict(xi=out, poses=torch.from_numpy(poses))
    wl = torch.tensor(proposal.LOSS_W, dtype=F64, device=DEV)
    outs, total = [], 0.0
    for c, t in zip(parts, xi.split(32)):
        out = _net64(c, p)
        loss = (wl * (out - t.double()) ** 2).sum() / case["batch"]
        loss.backward()
        outs.append(out.detach())
        total += float(loss.detach())
    g, st = p.grad, sd["step"] + 1
    m = 0.9 * sd["m"].to(DEV).double() + 0.1 * g
    v = 0.999 * sd["v"].to(DEV).double() + 0.001 * g * g
    q = p.detach() - LR * (m / (1 - 0.9 ** st)) / ((v / (1 - 0.999 ** st)).sqrt() + 1e-8)
    return dict(loss=torch.tensor([total], dtype=F64), out=torch.cat(outs), grads=g, params=q, m=m, v=v)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("propose", "train"):
        return _exact_net(case, seed)
    if kind in ("batch", "consistency"):
        # a hypothesis that ends in a wrong basin has no 64-bit value; the check's results are decisions
        return None
    w, prm = _world(case, seed), _params(case)
    if kind == "grid":
        poses = np.stack([_mul(_se3_exp(v), w.T0).reshape(12) for v in w.xi.double().cpu().numpy()])
        return dict(poses=torch.from_numpy(poses), scores=None, best=None, best_pose=None)
    if kind == "register":
        T, sums = _icp64(w.kp, w.depth, w.nw, w.sp, w.pix, w.nrm, w.T0, prm)
        return dict(pose=torch.from_numpy(T.reshape(12)), sums=sums, counts=None)
    if kind == "fuse":
        d, nw = _fuse64(w.kp, w.depth, w.nw, w.sp, w.pix, w.nrm, w.T0, prm)
        return dict(depth=d, nw=nw)
    depth, idx, xyz, has = _project64(w.scans[0], w.sp)
    nrm = _normals64(depth, xyz, has, w.sp, prm)
    if prm.atrous_levels:
        nrm = _atrous64(xyz, nrm, prm)
    pix = torch.cat([xyz, torch.ones_like(xyz[..., :1])], -1) * has[..., None]
    held = nrm.half() if w.f16 else nrm.float()
    T, sums = _icp64(w.kp, w.depth, w.nw, w.sp, pix, held, _mul(w.prev, w.motion), prm)
    kd, knw = _fuse64(w.kp, w.depth, w.nw, w.sp, pix, held, T, prm)
    return dict(pose=torch.from_numpy(T.reshape(12)), motion=torch.from_numpy(_mul(_inv(w.prev), T).reshape(12)),
                prev=torch.from_numpy(T.reshape(12)), sums=sums, counts=None, kf_depth=kd, kf_nw=knw,
                depth=torch.where(has, xyz.double().norm(dim=-1), torch.zeros_like(depth).double()), idx=None,
                pix=pix.double(), nrm=nrm)
