"""Performance cases of the surfel rasterizer: what a user's program calls,
through the package's public entry points.

Kinds (``case["kind"]``):
  render    bin + sort and forward of one frame (a viewer, a depth prediction)
  step      gradients zeroed, then one mapping step: bin + sort, forward with
            the loss, backward (``Rasterizer.step``); one map, 1 to 8 keyframes
  autograd  the same iteration through the autograd functions, the default
            driver of ``mapping.MappingWindow``
  maps      several maps of uneven size, one frame each, one captured call
            sequence replayed (``batched.BatchedMaps``)
  keyframe  new surfels from one scan's points (``keyframe.initialise``)
  manage    one map-management step that carries the optimiser's moments
            (``manage.MapManager.step``)
  track     trackable targets of a map (``track.trackable_targets``)
  adam      one fused Adam step of a map (``render.adam_step``)

Inputs are seeded simulations of a spinning LiDAR in a street (ground,
facades, boxes) or a room, generated on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_04127_gb300 import batched, keyframe, manage, mapping, render, scenes, track

GZ, FACADE_Y, FACADE_TOP = -1.8, 8.0, 10.2     # street: ground, facades (metres)
TILES = ((8, 8), (16, 16), (8, 32))


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # smallest call: a 2,000-surfel room seen once; latency and launches
        dict(name="room_render", kind="render", scene="room", n=2000, H=32, W=512, tile_h=16, tile_w=16, elev_deg=15.0,
             frames=1),
        # smallest mapping step, an odd frame whose last tiles are ragged
        dict(name="ragged_step", kind="step", scene="room", n=1500, H=37, W=100, tile_h=8, tile_w=8, elev_deg=30.0,
             frames=1),
        # ordinary frame of a 128-beam sensor: rendering alone
        dict(name="street_render", kind="render", scene="street", n=200_000, H=128, W=1024, tile_h=8, tile_w=8,
             elev_deg=45.0, frames=1),
        # ordinary mapping step, the benchmark's workload
        dict(name="street_step", kind="step", scene="street", n=200_000, H=128, W=1024, tile_h=8, tile_w=8,
             elev_deg=45.0, frames=1),
        # a 1M-surfel map against a window of 8 keyframes: the mapping loop of
        # a long sequence (dense maps: long tile lists)
        dict(name="window_step", kind="step", scene="track", n=1_000_000, H=128, W=1024, tile_h=8, tile_w=8,
             elev_deg=45.0, frames=8),
        # the default (autograd) driver on a small window
        dict(name="window_autograd", kind="autograd", scene="street", n=200_000, H=64, W=1024, tile_h=8, tile_w=8,
             elev_deg=45.0, frames=2),
        # several robots' maps in one captured step, the largest case
        dict(name="maps_graph", kind="maps", maps=6, n_min=50_000, n_max=2_000_000, tile_h=8, tile_w=8,
             elev_deg=45.0),
        # keyframe scans of a 64-beam and of a 128-beam sensor
        dict(name="keyframe_64", kind="keyframe", H=64, W=1024, elev_deg=45.0, k=20),
        dict(name="keyframe_128", kind="keyframe", H=128, W=1024, elev_deg=45.0, k=20),
        # map budget control of a 1M-surfel map that runs often: each pass
        # removes at most 1 % of the survivors
        dict(name="manage_1m", kind="manage", n=1_000_000),
        # what the tracker asks of a 1M-surfel map at every scan
        dict(name="track_1m", kind="track", n=1_000_000, keep=0.4),
        # the optimiser's part of a mapping iteration over 1M surfels
        dict(name="adam_1m", kind="adam", n=1_000_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "step", "step", "window", "autograd", "maps", "keyframe", "keyframe", "manage",
                       "manage", "track", "adam"])
    th, tw = rng.choice(TILES)
    if kind in ("render", "step"):
        room = rng.random() < 0.3
        return dict(kind=kind, scene="room" if room else "street", n=_log_int(rng, 1000, 20_000 if room else 250_000),
                    H=_log_int(rng, 24, 128), W=_log_int(rng, 96, 2048), tile_h=th, tile_w=tw,
                    elev_deg=round(rng.uniform(10.0, 45.0), 2), frames=1)
    if kind == "window":
        return dict(kind="step", scene="track", n=_log_int(rng, 100_000, 1_000_000), H=rng.choice([64, 100, 128]),
                    W=rng.choice([720, 1024, 1030]), tile_h=8, tile_w=8, elev_deg=45.0, frames=rng.randint(2, 8))
    if kind == "autograd":
        return dict(kind="autograd", scene="street", n=_log_int(rng, 20_000, 250_000), H=rng.choice([32, 64, 128]),
                    W=rng.choice([512, 900, 1024]), tile_h=th, tile_w=tw, elev_deg=round(rng.uniform(15.0, 45.0), 2),
                    frames=rng.randint(1, 3))
    if kind == "maps":
        return dict(kind="maps", maps=rng.randint(2, 6), n_min=_log_int(rng, 10_000, 60_000),
                    n_max=_log_int(rng, 100_000, 1_500_000), tile_h=8, tile_w=8, elev_deg=45.0)
    if kind == "keyframe":
        return dict(kind="keyframe", H=_log_int(rng, 16, 128), W=_log_int(rng, 300, 1100),
                    elev_deg=round(rng.uniform(15.0, 45.0), 2), k=rng.choice([8, 12, 20, 20, 20, 24, 32]))
    if kind == "manage":
        return dict(kind="manage", n=_log_int(rng, 20_000, 1_000_000))
    if kind == "track":
        return dict(kind="track", n=_log_int(rng, 10_000, 2_000_000), keep=round(rng.uniform(0.1, 0.9), 3))
    return dict(kind="adam", n=_log_int(rng, 10_000, 2_000_000))


# ---------------------------------------------------------------------------
# Seeded inputs (on the GPU)
# ---------------------------------------------------------------------------
DEV = "cuda"


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)


def _uni(g, shape, lo=0.0, hi=1.0):
    return torch.rand(shape, generator=g, device=DEV) * (hi - lo) + lo


def _boxes(g, x0, x1, clear_x):
    """Boxes with edges U(0.2, 1.5) m on the ground, 2,000 per 120 m of street,
    clear of the sensor positions: (lo [B,3], hi [B,3])."""
    m = int(2000 * (x1 - x0) / 120)
    c = torch.stack([_uni(g, (m,), x0, x1), _uni(g, (m,), -7.2, 7.2)], 1)
    e = _uni(g, (m, 3), 0.2, 1.5)
    cx = torch.tensor(clear_x, device=DEV)
    d = (c[:, :1] - cx[None]).abs().amin(1) - e[:, 0] / 2
    dy = c[:, 1].abs() - e[:, 1] / 2
    ok = (d > 2.5) | (dy > 2.5)
    c, e = c[ok], e[ok]
    z = torch.full_like(c[:, :1], GZ)
    return torch.cat([c - e[:, :2] / 2, z], 1), torch.cat([c + e[:, :2] / 2, z + e[:, 2:]], 1)


def _rays(H, W, elev_deg):
    em = math.radians(elev_deg)
    th = em - (torch.arange(H, device=DEV, dtype=torch.float32) + 0.5) * (2 * em / H)
    ph = (torch.arange(W, device=DEV, dtype=torch.float32) + 0.5) * (2 * math.pi / W)
    ct, st = torch.cos(th)[:, None], torch.sin(th)[:, None]
    return torch.stack([ct * torch.cos(ph), ct * torch.sin(ph), st.expand(H, W)], -1).reshape(-1, 3)


def _yaw(a):
    return torch.tensor([[math.cos(a), -math.sin(a), 0.0], [math.sin(a), math.cos(a), 0.0], [0.0, 0.0, 1.0]],
                        device=DEV)


def _take(t, n, tn, nn, ok):
    upd = ok & (tn > 1e-3) & (tn < t)
    return torch.where(upd, tn, t), torch.where(upd[:, None], nn, n)


def _cast(scene, o, d, boxes, max_range=150.0):
    """First hit of each ray: (t [M], inf on a miss; normal [M,3])."""
    t = torch.full((d.shape[0],), math.inf, device=DEV)
    n = torch.zeros_like(d)
    if scene == "room":
        for ax, lo, hi in ((0, -10.0, 10.0), (1, -10.0, 10.0), (2, -2.5, 2.5)):
            for plane, sgn in ((lo, 1.0), (hi, -1.0)):
                nn = torch.zeros(3, device=DEV)
                nn[ax] = sgn
                t, n = _take(t, n, (plane - o[ax]) / d[:, ax], nn.expand_as(d), torch.ones_like(t, dtype=torch.bool))
        return t, n
    t, n = _take(t, n, (GZ - o[2]) / d[:, 2], torch.tensor([0.0, 0.0, 1.0], device=DEV).expand_as(d), d[:, 2] < 0)
    for sgn in (1.0, -1.0):
        tf = (sgn * FACADE_Y - o[1]) / d[:, 1]
        t, n = _take(t, n, tf, torch.tensor([0.0, -sgn, 0.0], device=DEV).expand_as(d), o[2] + tf * d[:, 2] <= FACADE_TOP)
    lo, hi = boxes
    near = (lo[:, 0] - o[0]).abs() < 60.0
    lo, hi = lo[near] - o, hi[near] - o
    inv = 1.0 / torch.where(d.abs() > 1e-9, d, torch.full_like(d, 1e-9))
    step = max(1, (1 << 26) // max(1, d.shape[0]))
    for b in range(0, lo.shape[0], step):
        t_in = torch.full((d.shape[0], min(step, lo.shape[0] - b)), -math.inf, device=DEV)
        t_out = torch.full_like(t_in, math.inf)
        ax_in = torch.zeros_like(t_in, dtype=torch.int8)
        for ax in range(3):
            t0 = lo[None, b:b + step, ax] * inv[:, ax, None]
            t1 = hi[None, b:b + step, ax] * inv[:, ax, None]
            a, z = torch.minimum(t0, t1), torch.maximum(t0, t1)
            ax_in = torch.where(a > t_in, ax, ax_in)
            t_in, t_out = torch.maximum(t_in, a), torch.minimum(t_out, z)
        hit, at = torch.where((t_in <= t_out) & (t_in > 1e-3), t_in, math.inf).min(1)
        axis = ax_in.gather(1, at[:, None]).long()
        nn = torch.zeros_like(d).scatter_(1, axis, -torch.sign(d.gather(1, axis)))
        t, n = _take(t, n, hit, nn, torch.isfinite(hit))
    t = torch.where(t > max_range, math.inf, t)
    return t, n


def _scan(g, scene, boxes, x, yaw, H, W, elev_deg, noise=0.02, drop=0.1):
    """One simulated scan: range image D [H,W] (0 = no return), points and
    normals [HW,3] in the world, valid [HW], points in the sensor frame."""
    o = torch.tensor([x, 0.0, 0.0], device=DEV)
    ds = _rays(H, W, elev_deg)
    d = ds @ _yaw(yaw).T
    t, n = _cast(scene, o, d, boxes)
    r = t + noise * torch.randn(t.shape, generator=g, device=DEV)
    valid = torch.isfinite(t) & (torch.rand(t.shape, generator=g, device=DEV) >= drop) & (r > 0.3)
    r = torch.where(valid, r, 0.0)
    n = torch.where(((n * d).sum(1) > 0)[:, None], -n, n)
    return r.reshape(H, W), o + r[:, None] * d, n, valid, r[:, None] * ds


def _kappa(H, W, elev_deg):
    return 1.5 * max(2 * math.radians(elev_deg) / H, 2 * math.pi / W)


def _quats(g, n):
    """Unit quaternions whose third axis is n, with a random tangent."""
    q = torch.stack([1.0 + n[:, 2], -n[:, 1], n[:, 0], torch.zeros_like(n[:, 0])], 1)
    q = torch.where((n[:, 2:] < -0.9999).expand_as(q), torch.tensor([0.0, 1.0, 0.0, 0.0], device=DEV), q)
    q = q / q.norm(dim=1, keepdim=True)
    a = _uni(g, (n.shape[0],), 0.0, math.pi)
    c, s = torch.cos(a), torch.sin(a)
    w, x, y, z = q.unbind(1)
    return torch.stack([w * c - z * s, x * c + y * s, y * c - x * s, z * c + w * s], 1)


def _surfels(g, pts, nrm, rng_r, kappa, scale=None):
    n = pts.shape[0]
    if scale is None:
        sig = torch.stack([torch.ones(n, device=DEV), _uni(g, (n,), 0.4, 1.0)], 1)
        scale = (kappa * rng_r.clamp(min=1.0)[:, None] * sig).clamp(1e-3, 1.0)
    a = _uni(g, (n,), 0.3, 0.9)
    return [pts.contiguous(), _quats(g, nrm).contiguous(), torch.log(scale).contiguous(), torch.log(a / (1 - a))]


def _subset(g, k, n):
    return torch.sort(torch.randperm(k, generator=g, device=DEV)[:n]).values


def _frame(H, W, tile_h, tile_w, elev_deg, x, yaw):
    e = math.radians(elev_deg)
    return scenes.Frame(H, W, tile_h, tile_w, -e, e, scenes.pose_matrix(yaw, (x, 0.0, 0.0)))


def _target(D, nrm, valid):
    H, W = D.shape
    N = torch.where(valid[:, None], nrm, 0.0).T.reshape(3, H, W)
    return D.contiguous(), N.contiguous()


def _scene_inputs(case, seed):
    """(map tensors, frames, targets) of a render / step / autograd case."""
    g = _gen(seed)
    H, W, el, F, n = case["H"], case["W"], case["elev_deg"], case["frames"], case["n"]
    mk = lambda x, yaw: _frame(H, W, case["tile_h"], case["tile_w"], el, x, yaw)
    if case["scene"] == "room":
        # surfels on the six faces, scales U(5, 30) cm, 2 cm off the faces
        lo, hi = torch.tensor([-10.0, -10.0, -2.5], device=DEV), torch.tensor([10.0, 10.0, 2.5], device=DEV)
        p = _uni(g, (n, 3)) * (hi - lo) + lo
        face = torch.multinomial(torch.tensor([4.0, 4.0, 1.0, 1.0, 1.0, 1.0], device=DEV), n, replacement=True,
                                 generator=g)
        ax = torch.where(face < 2, 2, torch.where(face < 4, 0, 1))
        side = (face % 2).float()
        nrm = torch.zeros(n, 3, device=DEV).scatter_(1, ax[:, None], (1 - 2 * side)[:, None])
        off = 0.02 * torch.randn(n, generator=g, device=DEV)
        p = p.scatter(1, ax[:, None], (lo[ax] + side * (hi - lo)[ax] + (1 - 2 * side) * off)[:, None])
        params = _surfels(g, p, nrm, None, None, scale=_uni(g, (n, 2), 0.05, 0.30))
        D, _, tn, v, _ = _scan(g, "room", None, 0.0, 0.3, H, W, el, drop=0.0)
        return params, [mk(0.0, 0.3)], [_target(D, tn, v)]
    if case["scene"] == "street":
        # two (or more) merged scans, as a map built from scans is: in scan order
        xs = [1.5 * i for i in range(max(F, 2))]
        boxes = _boxes(g, -60.0, 60.0, xs)
        mh, mw = max(H, 128), max(W, 1024)
        scans = [_scan(g, "street", boxes, x, 0.3 + 0.1 * i, mh, mw, 45.0) for i, x in enumerate(xs)]
    else:
        # a 200 m track scanned every 3 m; keyframes 3 m apart in its middle
        xs = [-100.0 + 3.0 * i for i in range(67)]
        boxes = _boxes(g, -110.0, 110.0, xs)
        mh, mw = 64, 1024
        scans = [_scan(g, "street", boxes, x, 0.05 * i, mh, mw, 45.0) for i, x in enumerate(xs)]
    pts = torch.cat([s[1][s[3]] for s in scans])
    nrm = torch.cat([s[2][s[3]] for s in scans])
    r = torch.cat([s[4][s[3]].norm(dim=1) for s in scans])
    sel = _subset(g, pts.shape[0], n)
    params = _surfels(g, pts[sel], nrm[sel], r[sel], _kappa(mh, mw, 45.0))
    k0 = len(xs) // 2 - F // 2 if case["scene"] == "track" else 0
    frames, targets = [], []
    for j in range(F):
        yaw = 0.3 + 0.02 * j
        D, _, tn, v, _ = _scan(g, "street", boxes, xs[k0 + j], yaw, H, W, el)
        frames.append(mk(xs[k0 + j], yaw))
        targets.append(_target(D, tn, v))
    return params, frames, targets


def _surface_map(g, n, x, boxes):
    """n points uniform by area on the street within +-(20 + n / 25k) m of x:
    a map that many viewpoints built."""
    half = 20.0 + n / 25000.0
    lo, hi = boxes
    near = (lo[:, 0] >= x - half) & (hi[:, 0] <= x + half)
    lo, hi = lo[near], hi[near]
    e = hi - lo
    fa = torch.stack([e[:, 0] * e[:, 1], e[:, 1] * e[:, 2], e[:, 1] * e[:, 2], e[:, 0] * e[:, 2], e[:, 0] * e[:, 2]], 1)
    area = torch.tensor([2 * FACADE_Y * 2 * half, 4 * half * (FACADE_TOP - GZ), float(fa.sum())], device=DEV)
    kind = torch.multinomial(area, n, replacement=True, generator=g)
    px = _uni(g, (n,), x - half, x + half)
    side = torch.where(torch.rand(n, generator=g, device=DEV) < 0.5, -1.0, 1.0)
    z = torch.zeros(n, device=DEV)
    ground = torch.stack([px, _uni(g, (n,), -FACADE_Y, FACADE_Y), z + GZ], 1)
    facade = torch.stack([px, side * FACADE_Y, _uni(g, (n,), GZ, FACADE_TOP)], 1)
    face = torch.multinomial(fa.reshape(-1), n, replacement=True, generator=g)
    b, f = face // 5, face % 5
    u = lo[b] + _uni(g, (n, 3)) * e[b]
    ax = torch.where(f == 0, 2, torch.where(f < 3, 0, 1))
    up = (f == 0) | (f == 2) | (f == 4)
    u = u.scatter(1, ax[:, None], torch.where(up, hi[b].gather(1, ax[:, None])[:, 0], lo[b].gather(1, ax[:, None])[:, 0])[:, None])
    bn = torch.zeros(n, 3, device=DEV).scatter_(1, ax[:, None], torch.where(up, 1.0, -1.0)[:, None])
    k = kind[:, None]
    pts = torch.where(k == 0, ground, torch.where(k == 1, facade, u))
    nrm = torch.where(k == 0, torch.tensor([0.0, 0.0, 1.0], device=DEV),
                      torch.where(k == 1, torch.stack([z, -side, z], 1), bn))
    view = torch.tensor([x, 0.0, 0.0], device=DEV) - pts
    return pts, torch.where(((nrm * view).sum(1) < 0)[:, None], -nrm, nrm), view.norm(dim=1)


def _map_sizes(case):
    m = case["maps"]
    r = (case["n_max"] / case["n_min"]) ** (1.0 / max(1, m - 1))
    return [int(round(case["n_min"] * r ** i)) for i in range(m)]


def _numpy_map(p):
    return scenes.Surfels(*[t.cpu().numpy() for t in p])


def _numpy_targets(targets):
    return [scenes.Target(D.cpu().numpy(), N.cpu().numpy()) for D, N in targets]


def _maps_inputs(case, seed):
    g = _gen(seed)
    sizes = _map_sizes(case)
    shapes = [(64, 1024), (128, 1024), (128, 2048)]
    span = 20.0 + max(sizes) / 25000.0
    xs = [25.0 * i for i in range(len(sizes))]
    boxes = _boxes(g, xs[0] - span - 10, xs[-1] + span + 10, xs)
    maps, frames, targets = [], [], []
    for i, (n, x) in enumerate(zip(sizes, xs)):
        H, W = shapes[i % 3]
        pts, nrm, r = _surface_map(g, n, x, boxes)
        maps.append(_numpy_map(_surfels(g, pts, nrm, r, _kappa(H, W, case["elev_deg"]))))
        D, _, tn, v, _ = _scan(g, "street", boxes, x, 0.1 * i, H, W, case["elev_deg"])
        frames.append(_frame(H, W, case["tile_h"], case["tile_w"], case["elev_deg"], x, 0.1 * i))
        targets.append(_target(D, tn, v))
    return maps, frames, _numpy_targets(targets)


def _keyframe_inputs(case, seed):
    g = _gen(seed)
    boxes = _boxes(g, -60.0, 60.0, [0.0])
    _, _, _, v, ps = _scan(g, "street", boxes, 0.0, 0.3, case["H"], case["W"], case["elev_deg"], drop=0.0)
    ps = ps[v]                                       # in scan order, random drops down to the usual share
    return ps[_subset(g, ps.shape[0], _keyframe_n(case))].contiguous(), \
        scenes.pose_matrix(0.3, (12.0, -3.0, 0.5)).astype(np.float64)


def _keyframe_n(case):
    return int(0.78 * case["H"] * case["W"])


def _long_map(seed, n):
    """A map of n surfels along a street, in chunks of 25 m, with its points'
    distance to their sensor."""
    g = _gen(seed)
    half = 20.0 + n / 25000.0
    boxes = _boxes(g, -half - 10, half + 10, [0.0])
    pts, nrm, r = _surface_map(g, n, 0.0, boxes)
    order = torch.argsort(torch.floor(pts[:, 0] / 25.0), stable=True)
    pts, nrm = pts[order] + 0.02 * torch.randn(n, 3, generator=g, device=DEV), nrm[order]
    return g, _surfels(g, pts, nrm, (r[order] % 60.0), 0.0184)


def _manage_inputs(case, seed):
    """A map with its tracking signals: covariance eigenvalues of planar
    (most), linear and scattered neighbourhoods, and exponential residuals."""
    n = case["n"]
    g, params = _long_map(seed, n)
    # opacity logits: the quantiles of N(0.5, 1.5), shuffled
    rank = (torch.randperm(n, generator=g, device=DEV).double() + 0.5) / n
    params[3] = (0.5 + 1.5 * math.sqrt(2.0) * torch.erfinv(2.0 * rank - 1.0)).float()
    kind = torch.rand(n, generator=g, device=DEV)[:, None]
    ratio = torch.where(kind < 0.75, torch.tensor([1.0, 0.7, 0.002], device=DEV),
                        torch.where(kind < 0.9, torch.tensor([1.0, 0.05, 0.01], device=DEV),
                                    torch.tensor([1.0, 0.6, 0.3], device=DEV)))
    lam = (ratio * _uni(g, (n, 3), 0.6, 1.4) * _uni(g, (n, 1), 0.002, 0.05)).contiguous()
    res = -0.02 * torch.log1p(-torch.rand(n, generator=g, device=DEV))
    moments = [torch.randn(n, 10, generator=g, device=DEV) * 1e-3,
               torch.rand(n, 10, generator=g, device=DEV) * 1e-6]
    return params, lam, res, moments


def _track_inputs(case, seed):
    n = case["n"]
    g, params = _long_map(seed, n)
    sel = torch.randperm(n, generator=g, device=DEV) < _track_n(case)
    # the others are untrackable, not seen for long, or too faint
    why = torch.where(sel, -1, torch.randint(0, 3, (n,), generator=g, device=DEV))
    mask = (why != 0).to(torch.uint8)
    last = torch.where(why == 1, torch.randint(0, 3, (n,), generator=g, device=DEV),
                       torch.randint(3, 12, (n,), generator=g, device=DEV)).to(torch.int32)
    a = torch.where(why == 2, _uni(g, (n,), 0.3, 0.49), _uni(g, (n,), 0.51, 0.9))
    params[3] = torch.log(a / (1 - a))
    return params, mask, last


def _track_n(case):
    return max(1, int(case["keep"] * case["n"]))


def _adam_inputs(case, seed):
    n = case["n"]
    g, params = _long_map(seed, n)
    seen = (torch.rand(n, generator=g, device=DEV) < 0.6).float()   # surfels no frame saw have no gradient
    grads = [1e-3 * torch.randn(t.shape, generator=g, device=DEV) * (seen if t.dim() == 1 else seen[:, None])
             for t in params]
    return params, grads, 1e-3 * torch.randn(10 * n, generator=g, device=DEV), \
        1e-6 * torch.rand(10 * n, generator=g, device=DEV)


LR = mapping.DEFAULT_LR
ADAM_STEP = 7


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("render", "step"):
        params, frames, targets = _scene_inputs(case, seed)
        rast = render.Rasterizer(frames)
        rast.bin_sort([params], check=True)          # sizes the workspace, as a mapping loop's first step does
        return dict(kind=kind, params=params, rast=rast, targets=targets, grads=[torch.zeros_like(p) for p in params])
    if kind == "autograd":
        params, frames, targets = _scene_inputs(case, seed)
        win = mapping.MappingWindow(_numpy_map(params), frames, _numpy_targets(targets))
        return dict(kind=kind, win=win)
    if kind == "maps":
        maps, frames, targets = _maps_inputs(case, seed)
        B = batched.BatchedMaps(maps, frames, targets)
        B.capture()
        return dict(kind=kind, B=B)
    if kind == "keyframe":
        pts, pose = _keyframe_inputs(case, seed)
        return dict(kind=kind, pts=pts, pose=pose, p=keyframe.params(k=case["k"]))
    if kind == "manage":
        params, lam, res, moments = _manage_inputs(case, seed)
        return dict(kind=kind, params=params, lam=lam, res=res, moments=moments, mgr=manage.MapManager(),
                    p=manage.params(prune_cap=0.01))
    if kind == "track":
        params, mask, last = _track_inputs(case, seed)
        return dict(kind=kind, params=params, mask=mask, last=last)
    params, grads, m, v = _adam_inputs(case, seed)
    return dict(kind=kind, params=params, grads=grads, m=m, v=v)


def run(s):
    kind = s["kind"]
    if kind == "render":
        S = s["rast"].bin_sort([s["params"]], check=False)
        return [dict(A=o.A, S_t=o.S_t, S_n=o.S_n, T_final=o.T_final, n_contrib=o.n_contrib)
                for o in s["rast"].forward([s["params"]], S)]
    if kind == "step":
        for g in s["grads"]:
            g.zero_()
        return dict(loss=s["rast"].step([s["params"]], s["targets"], [s["grads"]]), grads=s["grads"])
    if kind == "autograd":
        loss, grads = s["win"].loss_and_grads()
        return dict(loss=loss, grads=grads)
    if kind == "maps":
        s["B"].replay()
        return dict(loss=s["B"].rast.loss_out, grads=s["B"].grads)
    if kind == "keyframe":
        out = keyframe.initialise(s["pts"], s["pose"], s["p"])
        return {k: out[k] for k in ("mean", "quat", "log_scale", "logit", "lam", "u", "knn")}
    if kind == "manage":
        new, carried, info = s["mgr"].step(s["params"], s["lam"], s["res"], s["p"], carry=s["moments"])
        return dict(map=new, moments=carried, score=info["score"], src=info["src"], role=info["role"],
                    counts=list(info["counts"]))
    if kind == "track":
        return list(track.trackable_targets(s["params"], s["mask"], s["last"], 3, 0.5))
    render.adam_step(s["params"], s["grads"], s["m"], s["v"], ADAM_STEP, lr=LR)
    return dict(params=s["params"], grads=s["grads"], m=s["m"], v=s["v"])


# ---------------------------------------------------------------------------
# Work a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: every input read and every output written once.  FLOPs of the
    compositing: about 50 composited pairs per pixel, 39 each forward (plane
    intersection, Gaussian, sums) and 97 more backward; of the k-NN: 8 per
    distance, each point against the 3k points around it."""
    kind = case["kind"]
    if kind in ("render", "step", "autograd"):
        px = case["H"] * case["W"] * case["frames"]
        if kind == "render":
            return dict(bytes=40 * case["n"] + 28 * px, flops=50 * 39 * px)
        return dict(bytes=80 * case["n"] + 16 * px, flops=50 * 136 * px)
    if kind == "maps":
        shapes = [(64, 1024), (128, 1024), (128, 2048)]
        px = sum(shapes[i % 3][0] * shapes[i % 3][1] for i in range(case["maps"]))
        return dict(bytes=80 * sum(_map_sizes(case)) + 16 * px, flops=50 * 136 * px)
    if kind == "keyframe":
        n = _keyframe_n(case)
        return dict(bytes=n * (12 + 40 + 16 + 4 * case["k"]), flops=8 * 3 * case["k"] * n)
    n = case["n"]
    if kind == "manage":
        return dict(bytes=n * (40 + 16 + 4 + 45 + 2 * 80), flops=40 * n)
    if kind == "track":
        sel = _track_n(case)
        return dict(bytes=9 * n + sel * (36 + 44), flops=60 * sel)
    return dict(bytes=10 * n * 32, flops=10 * n * 14)


# ---------------------------------------------------------------------------
# 64-bit results
# ---------------------------------------------------------------------------
def _axes64(q):
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    tu = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + w * z), 2 * (x * z - w * y)], 1)
    tv = torch.stack([2 * (x * y - w * z), 1 - 2 * (x * x + z * z), 2 * (y * z + w * x)], 1)
    nn = torch.stack([2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y)], 1)
    return tu, tv, nn


def _depth_keys(mean, pose32):
    """The binary32 |mu_sensor| that orders the surfels, one rounding per
    operation in the order of its definition."""
    R, o = pose32[:, :3], pose32[:, 3]
    d = [mean[:, k] - o[k] for k in range(3)]
    c = [(R[0, k] * d[0] + R[1, k] * d[1]) + R[2, k] * d[2] for k in range(3)]
    return torch.sqrt((c[0] * c[0] + c[1] * c[1]) + c[2] * c[2])


def _render64(params, frames, targets, loss):
    """Planes per frame, and (with targets) the loss vector and gradients."""
    P64 = [p.detach().double().requires_grad_(targets is not None) for p in params]
    planes, terms, F = [], [], len(frames)
    for fi, fr in enumerate(frames):
        H, W = fr.H, fr.W
        pose32 = torch.from_numpy(np.asarray(fr.pose, np.float32).reshape(3, 4)).to(DEV)
        pose = pose32.double()
        R, o = pose[:, :3], pose[:, 3]
        tu, tv, nn = _axes64(P64[1])
        full = [(P64[0] - o) @ R, tu @ R, tv @ R, nn @ R, torch.exp(P64[2]), torch.sigmoid(P64[3])]
        leaf = [t.detach().requires_grad_(targets is not None) for t in full]
        with torch.no_grad():
            key = _depth_keys(params[0], pose32)
            order = torch.sort(key, stable=True).indices      # ties by index
            mu = leaf[0][order]
            r = mu.norm(dim=1)
            rho = 3.001 * leaf[4][order].amax(1)
            cap = torch.where(r > rho, torch.asin((rho / r).clamp(max=1.0)), math.pi)
            mdir = mu / r[:, None]
        emin, emax = float(np.float32(fr.elev_min)), float(np.float32(fr.elev_max))
        th = emax - (torch.arange(H, device=DEV, dtype=torch.float64) + 0.5) * ((emax - emin) / H)
        ph = (2 * torch.arange(W, device=DEV, dtype=torch.float64) + 1) * math.pi / W
        rays = torch.stack([torch.cos(th)[:, None] * torch.cos(ph), torch.cos(th)[:, None] * torch.sin(ph),
                            torch.sin(th)[:, None].expand(H, W)], -1)
        out = torch.zeros(6, H, W, device=DEV, dtype=torch.float64)
        if targets is not None:
            D, N = targets[fi][0].double(), targets[fi][1].double()
            mD = D > 0
            mN = mD & ((N * N).sum(0) > 0)
            nD, nN = max(int(mD.sum()), 1), max(int(mN.sum()), 1)
            acc = [torch.zeros((), device=DEV, dtype=torch.float64) for _ in range(3)]
        bh, bw = 8, 32
        for r0 in range(0, H, bh):
            for c0 in range(0, W, bw):
                d = rays[r0:r0 + bh, c0:c0 + bw].reshape(-1, 3)
                with torch.no_grad():
                    ctr = d.mean(0)
                    ctr = ctr / ctr.norm()
                    half = torch.acos((d @ ctr).clamp(-1.0, 1.0)).max() + 1e-4
                    idx = order[torch.acos((mdir @ ctr).clamp(-1.0, 1.0)) <= cap + half]
                m_, u_, v_, n_, s_, al = [t[idx] for t in leaf]
                den = d @ n_.T
                t = (n_ * m_).sum(1)[None] / torch.where(den.abs() >= 1e-6, den, torch.ones_like(den))
                u = (t * (d @ u_.T) - (u_ * m_).sum(1)) / s_[:, 0]
                v = (t * (d @ v_.T) - (v_ * m_).sum(1)) / s_[:, 1]
                q = u * u + v * v
                a = (al * torch.exp(-0.5 * q)).clamp(max=0.99)
                ok = (den.abs() >= 1e-6) & (t > 0.2) & (q <= 9.0) & (a >= 1.0 / 255.0)
                a = torch.where(ok, a, 0.0)
                lT = torch.cumsum(torch.log1p(-a), 1)
                keep = lT >= math.log(1e-4)
                w = torch.where(keep, a * torch.exp(lT - torch.log1p(-a)), 0.0)
                A = w.sum(1)
                t = torch.where(ok, t, 0.0)
                St = (w * t).sum(1)
                Sn = (-(w * torch.sign(den.detach()))) @ n_
                Tf = torch.exp(torch.where(keep, torch.log1p(-a), 0.0).sum(1))
                shp = (min(bh, H - r0), min(bw, W - c0))
                with torch.no_grad():
                    out[:, r0:r0 + bh, c0:c0 + bw] = torch.cat([A[None], St[None], Sn.T, Tf[None]]).reshape(6, *shp)
                if targets is None:
                    continue
                Dm, Nm = D[r0:r0 + bh, c0:c0 + bw].reshape(-1), N[:, r0:r0 + bh, c0:c0 + bw].reshape(3, -1).T
                k, kn = mD[r0:r0 + bh, c0:c0 + bw].reshape(-1), mN[r0:r0 + bh, c0:c0 + bw].reshape(-1)
                Ld = torch.where(k, (St / (A + 1e-6) - Dm).abs(), 0.0).sum() / nD
                La = torch.where(k, -torch.log(A + 1e-6), 0.0).sum() / nD
                Nh = Sn / torch.sqrt((Sn * Sn).sum(1, keepdim=True) + 1e-12)
                Ln = torch.where(kn, 1.0 - (Nh * Nm).sum(1), 0.0).sum() / nN
                L = (Ld + loss.lambda_alpha * La + loss.lambda_n * loss.lambda_ng * Ln) / F
                if L.requires_grad and idx.numel():
                    L.backward()
                for j, x in enumerate((Ld, La, Ln)):
                    acc[j] += x.detach()
        planes.append(out)
        if targets is not None:
            terms.append(acc)
            torch.autograd.backward([f for f, l in zip(full, leaf) if l.grad is not None],
                                    [l.grad for l in leaf if l.grad is not None])
    if targets is None:
        return planes, None, None
    sm = torch.exp(P64[2]).amax(1)
    reg = loss.lambda_s * (sm - loss.s_max).clamp(min=0.0).sum()
    if float(reg.detach()) > 0.0:
        reg.backward()
    L = sum((a[0] + loss.lambda_alpha * a[1] + loss.lambda_n * loss.lambda_ng * a[2]) / F for a in terms) + reg.detach()
    vec = [L]
    for a in terms:
        vec += [*a, torch.zeros_like(L)]
    vec.append(L)
    return planes, torch.stack(vec), [p.grad if p.grad is not None else torch.zeros_like(p) for p in P64]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("render", "step", "autograd"):
        if case["n"] > 300_000 or case["H"] * case["W"] * case["frames"] > 300_000:
            return None                              # minutes in 64 bits
        params, frames, targets = _scene_inputs(case, seed)
        loss = render.LossParams()
        if kind == "render":
            with torch.no_grad():
                planes, _, _ = _render64(params, frames, None, loss)
            return [dict(A=o[0], S_t=o[1], S_n=o[2:5], T_final=o[5], n_contrib=None) for o in planes]
        _, vec, grads = _render64(params, frames, targets, loss)
        return dict(loss=vec if kind == "step" else vec[0], grads=grads)
    if kind == "keyframe":
        pts, pose = _keyframe_inputs(case, seed)
        p = keyframe.params(k=case["k"])
        x = pts.double()
        n, k = x.shape[0], case["k"]
        nb = torch.empty(n, k, dtype=torch.long, device=DEV)
        for a in range(0, n, 512):
            d = torch.zeros(min(512, n - a), n, device=DEV, dtype=torch.float64)
            for ax in range(3):
                d += (x[a:a + 512, ax, None] - x[None, :, ax]) ** 2
            nb[a:a + 512] = torch.topk(d, k, dim=1, largest=False).indices
        c = x[nb] - x[nb].mean(1, keepdim=True)
        c = c.cpu().numpy()
        lam, vec = np.linalg.eigh(np.einsum("nki,nkj->nij", c, c) / k)
        lam = torch.from_numpy(np.maximum(lam[:, ::-1], 0.0).copy()).to(DEV)
        nrm = torch.from_numpy(vec[:, :, 0].copy()).to(DEV)
        r = x.norm(dim=1)
        sig = torch.sqrt(lam)
        t1 = torch.where(sig[:, 0] > 0, sig[:, 1] / sig[:, 0], 1.0)
        s = p.kappa * r.clamp(min=1.0)[:, None] * torch.stack([torch.ones_like(t1), t1], 1)
        cosv = ((nrm * x).sum(1) / r).abs()
        u = torch.exp(-(r / p.r0) ** 2) * ((cosv - p.c0) / (1 - p.c0 + p.eps)).clamp(0.0, 1.0)
        al = p.alpha_min + (p.alpha_max - p.alpha_min) * u
        P = torch.from_numpy(np.asarray(pose, np.float64).reshape(3, 4)).to(DEV)
        return dict(mean=x @ P[:, :3].T + P[:, 3], quat=None, log_scale=torch.log(s.clamp(p.s_min, p.s_max)),
                    logit=torch.log(al / (1 - al)), lam=lam, u=u, knn=None)
    if kind == "manage":
        _, lam, res, _ = _manage_inputs(case, seed)
        p = manage.params()
        l = torch.sort(lam.double(), dim=1, descending=True).values
        rq = torch.sort(res).values[int(math.floor(p.q_res * (case["n"] - 1)))].double()
        lin = (l[:, 0] - l[:, 1]) / (l[:, 0] + p.eps)
        cur = (3 * l[:, 2] / (l.sum(1) + p.eps)).clamp(max=1.0)
        c = p.w_l * lin + p.w_c * cur + p.w_r * (res.double() / (rq + p.eps)).clamp(max=1.0)
        return dict(map=None, moments=None, score=c.clamp(0.0, 1.0), src=None, role=None, counts=None)
    if kind == "track":
        params, mask, last = _track_inputs(case, seed)
        i = torch.nonzero((mask != 0) & (last >= 3) & (params[3] >= 0.0))[:, 0]
        tu, tv, nn = _axes64(params[1][i].double())
        s = torch.exp(params[2][i].double())
        cov = sum(w[:, None, None] * e[:, :, None] * e[:, None, :]
                  for w, e in ((s[:, 0] ** 2, tu), (s[:, 1] ** 2, tv), (torch.full_like(s[:, 0], 0.01 ** 2), nn)))
        so = torch.sort(s, dim=1, descending=True).values
        kap = so[:, 0] / (so[:, 1] + 1e-6)
        lo, hi = kap.min(), kap.max()
        bar = (kap - lo) / (hi - lo) if float(hi) > float(lo) else torch.zeros_like(kap)
        ij = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
        return [None, params[0][i].double(), torch.stack([cov[:, a, b] for a, b in ij], 1),
                (1.0 / (bar + 1e-6)).clamp(max=10.0)]
    if kind == "adam":
        params, grads, m, v = _adam_inputs(case, seed)
        n = case["n"]
        g = torch.cat([x.double().reshape(-1) for x in grads])
        b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
        m = b1 * m.double() + (1 - b1) * g
        v = b2 * v.double() + (1 - b2) * g * g
        up = (m / (1 - b1 ** ADAM_STEP)) / (torch.sqrt(v / (1 - b2 ** ADAM_STEP)) + 1e-15)
        new, off = [], 0
        for x, lr in zip(params, LR):
            new.append(x.double() - lr * up[off:off + x.numel()].reshape(x.shape))
            off += x.numel()
        return dict(params=new, grads=[torch.zeros_like(x).double() for x in grads], m=m, v=v)
    return None
