"""The work that a program using this library has it do, as measurable cases.

Each case is one pass through the public Python entry points
(``engine.Scene``, ``engine.Batch``, ``engine.channel_correlation``,
``autograd.field``) on the seeded scenes of this repository (toy, district,
city, uneven batch), whose static geometry is the program's plan and whose
poses (vehicles, receivers) are drawn from the seed.

Operations
  host_frame   poses in host arrays: update, trace, fields, the call that
               waits and reports errors, received power read back (the loop of
               a first program or a notebook)
  frame        poses on the device: update, full retrace, fields (plain method;
               with static_cache, the refresh frame of the cached method)
  cached       update, low-density rediscovery into the previous frame's path
               cache with its revalidation, fields (cached method)
  fields       fields and statistics of a path set at several frequencies
  gradient     received-power loss, its gradient in the material parameters
               and transmitter positions
  revalidate   a path cache carried to the next frame, invalid paths removed
  backward     discovery from a subset of the receivers
  schedule     update and the per-receiver re-discovery schedule
  batch        update and batched retrace of scenes of uneven size
  correlation  Eq. 1 over a series of frames for every pair
"""
import functools
import math

import numpy as np
import torch

from paper_2303_10521_gb300 import autograd, engine, scenes

POSES = ("veh_pos", "veh_vel", "rx_pos", "rx_vel", "tx_pos", "tx_vel")


def listed():
    return [
        # the smallest program: 1 transmitter, 16 receivers, 20 buildings;
        # latency, launches and host copies count
        dict(name="toy_host_frame", op="host_frame", scene="toy", n_rays=100_000, depth=2),
        # the district workload, every frame retraced: 2 Tx, 1000 Rx, 200 vehicles
        dict(name="district_frame", op="frame", scene="district", n_rays=1_000_000, depth=3,
             n_veh=200, n_rx=1000, freqs=1, static_cache=False),
        # the benchmark frame: 2x2 km, 4 Tx x 1e7 rays, 10k Rx, 5000 vehicles
        dict(name="city_frame", op="frame", scene="city", blocks=40, n_rays=10_000_000, depth=4,
             n_veh=5000, n_rx=10_000, freqs=2, static_cache=False),
        # a refresh frame of the cached method on a part of the city, odd sizes
        dict(name="quarter_refresh_frame", op="frame", scene="city", blocks=19,
             n_rays=2_500_003, depth=4, n_veh=1237, n_rx=2501, freqs=2, static_cache=True),
        # the ordinary frame of the cached method on the benchmark city
        dict(name="city_cached_frame", op="cached", scene="city", blocks=40, n_rays=10_000_000,
             depth=4, n_veh=5000, n_rx=10_000, freqs=2, static_cache=True),
        # the same on the district without the static-hit cache
        dict(name="district_cached_frame", op="cached", scene="district", n_rays=1_000_000,
             depth=3, n_veh=200, n_rx=1000, freqs=1, static_cache=False),
        # another carrier or other materials on a path set already traced
        dict(name="city_fields", op="fields", scene="city", blocks=40, n_rays=10_000_000, depth=4,
             n_veh=5000, n_rx=10_000, freqs=2),
        # calibration of materials and transmitter positions
        dict(name="district_gradient", op="gradient", scene="district", n_rays=1_000_000, depth=3,
             n_veh=200, n_rx=1000),
        # a re-discovery of the due receivers only
        dict(name="city_backward", op="backward", scene="city", blocks=40, n_rays=50_000, depth=4,
             n_veh=5000, n_rx=10_000, n_ids=256),
        # which receivers are due: update and line of sight of every pair
        dict(name="city_schedule", op="schedule", scene="city", blocks=40, n_veh=5000,
             n_rx=10_000),
        # scenario sweep: 12 scenes of uneven size
        dict(name="uneven_batch", op="batch", n=12),
        # 300 frames of every pair of the city, 5 s of lags
        dict(name="city_correlation", op="correlation", frames=300, pairs=40_000, lag=50),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["host_frame", "frame", "frame", "cached", "cached", "fields", "gradient",
                     "revalidate", "backward", "schedule", "batch", "correlation"])
    if op == "host_frame":
        return dict(op=op, scene="toy", n_rays=_log(rng, 20_000, 1_000_000),
                    depth=rng.randint(1, 4))
    if op == "batch":
        return dict(op=op, n=rng.randint(4, 12))
    if op == "correlation":
        return dict(op=op, frames=rng.randint(50, 300), pairs=_log(rng, 100, 40_000),
                    lag=rng.randint(5, 50))
    if rng.random() < 0.5:
        c = dict(op=op, scene="district", n_rays=_log(rng, 100_000, 2_000_000),
                 depth=rng.randint(2, 4), n_veh=_log(rng, 10, 500), n_rx=_log(rng, 50, 4000))
    else:
        c = dict(op=op, scene="city", blocks=rng.randint(8, 40),
                 n_rays=_log(rng, 500_000, 8_000_000), depth=rng.randint(2, 4),
                 n_veh=_log(rng, 50, 5000), n_rx=_log(rng, 100, 10_000))
    if op in ("frame", "cached"):
        c.update(freqs=rng.randint(1, 2), static_cache=rng.random() < 0.5)
    elif op == "fields":
        c.update(freqs=rng.randint(1, 4))
    elif op == "revalidate":
        c.update(keep=rng.random() < 0.5)
    elif op == "backward":
        c.update(n_rays=_log(rng, 10_000, 60_000), n_ids=min(c["n_rx"], _log(rng, 4, 400)))
    elif op == "schedule":
        del c["n_rays"], c["depth"]
    return c


# ---------------------------------------------------------------------------
# inputs
@functools.lru_cache(maxsize=4)
def _desc(kind, blocks, n_veh, n_rx, n_rays, depth):
    if kind == "district":
        return scenes.district_scene(n_rays=n_rays, depth=depth, n_veh=n_veh, n_rx=n_rx)
    return scenes.city_scene(n_rays=n_rays, depth=depth, n_veh=n_veh, n_rx=n_rx, blocks=blocks)


@functools.lru_cache(maxsize=2)
def _batch_descs(n):
    return scenes.batched_scenes(seed=0, n=n)


def _scene_desc(case):
    return _desc(case["scene"], case.get("blocks", 0), case["n_veh"], case["n_rx"],
                 case.get("n_rays", 100_000), case.get("depth", 4))


def _on_device(frame):
    return scenes.Frame(*(torch.as_tensor(getattr(frame, f)).cuda() for f in POSES))


def _freqs(n):
    return [3.5e9, 28e9, 0.7e9, 6.0e9][:n]


def _paths(capacity):
    p = engine.Paths(capacity, "cuda")
    p.rec.zero_()
    return p


def _channel_outs(n, capacity, n_tx, n_rx):
    z = functools.partial(torch.zeros, dtype=torch.float64, device="cuda")
    return [engine.ChannelResult(z((capacity, 4)), z((n_tx, n_rx, 8)), z((n_rx, 2)))
            for _ in range(n)]


def _stack(chs):
    return [[c.path, c.pair, c.rx] for c in chs]


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    op = case["op"]
    S = dict(case=dict(case))
    if op == "host_frame":
        d = scenes.toy_scene(seed=int(seed), n_rays=case["n_rays"], depth=case["depth"])
        g, fr = engine.Scene(d), d.frame(0)
        capacity = max(4096, 8 * g.max_tx * g.max_rx)
        S.update(scene=g, frame=fr, freq=d.freqs[0], out=_paths(capacity),
                 chs=_channel_outs(1, capacity, g.max_tx, g.max_rx))
        return S
    if op == "correlation":
        S.update(h=_series(case, seed), lag=case["lag"])
        return S
    if op == "batch":
        descs = _batch_descs(case["n"])
        frames = [_on_device(d.frame(float(rng.uniform(0, 300)))) for d in descs]
        gs = [engine.Scene(d) for d in descs]
        for g, f in zip(gs, frames):
            g.update(f)
        b = engine.Batch(gs)
        for o in b.outs:
            o.rec.zero_()
        S.update(scenes=gs, frames=frames, batch=b)
        return S
    d = _scene_desc(case)
    k = float(rng.uniform(0, d.n_frames))
    before, now = _on_device(d.frame(k)), _on_device(d.frame(k + 1.0))
    g = engine.Scene(d)
    g.update(before)
    S.update(scene=g, frame=now)
    capacity = max(4096, 8 * g.n_tx * g.n_rx)
    if op == "frame":
        S.update(out=_paths(capacity), static=case["static_cache"], freqs=_freqs(case["freqs"]))
        if S["static"]:  # the frame before has filled the static-hit cache
            g.trace_async(S["out"], static_cache=True)
            g.sync()
            S["out"].rec.zero_()
        S["chs"] = _channel_outs(case["freqs"], capacity, g.n_tx, g.n_rx)
    elif op == "cached":
        static = case["static_cache"]
        kept = _paths(capacity)
        g.trace_async(kept, static_cache=static)
        g.sync()
        n_low = max(1, d.n_rays // 10)
        g.rediscover(kept, n_rays=n_low, static_cache=static, revalidate=True)
        g.sync()
        S.update(kept=kept, cache=_paths(capacity), n_low=n_low, static=static,
                 freqs=_freqs(case["freqs"]),
                 chs=_channel_outs(case["freqs"], capacity, g.n_tx, g.n_rx))
    elif op in ("fields", "gradient", "revalidate"):
        if op != "revalidate":
            g.update(now)
        found = _paths(capacity)
        g.trace_async(found)
        g.sync()
        S["paths"] = found
        if op == "fields":
            S.update(freqs=_freqs(case["freqs"]),
                     chs=_channel_outs(case["freqs"], capacity, g.n_tx, g.n_rx))
        elif op == "gradient":
            S.update(_calibration(d, g, found, rng))
        else:
            g.update(now)
            S.update(keep=case["keep"], cache=_paths(capacity))
    elif op == "backward":
        g.update(now)
        ids = np.sort(rng.choice(case["n_rx"], case["n_ids"], replace=False)).astype(np.int32)
        S.update(out=_paths(capacity), ids=torch.as_tensor(ids).cuda())
    elif op == "schedule":
        sched = engine.RefreshSchedule(g.n_tx, g.n_rx, "cuda", 3.5e9, d.dt)
        g.refresh_schedule(sched)
        S["sched"] = sched
    return S


def _calibration(d, g, found, rng):
    """Measured received power: the model's at perturbed materials, with 3 dB
    of measurement noise; the parameters start at the table's values."""
    t64 = functools.partial(torch.as_tensor, dtype=torch.float64, device="cuda")
    h = g.channel(found, d.freqs[0]).pair[..., :2]
    p = d.tx_power_w * (h ** 2).sum(-1).sum(0)
    mask = p > 0
    noise = t64(rng.normal(0, 3, g.n_rx))
    target = torch.where(mask, 10 * torch.log10(torch.where(mask, p, torch.ones_like(p)) * 1e3)
                         + noise, torch.zeros_like(p))
    return dict(eps=t64(d.eps_r * rng.uniform(0.95, 1.05, 8)).requires_grad_(),
                sig=t64(d.sigma * rng.uniform(0.95, 1.05, 8)).requires_grad_(),
                tx=g._frame["tx_pos"].double().requires_grad_(), mask=mask, target=target,
                power=d.tx_power_w, freq=d.freqs[0])


def _series(case, seed):
    """Coherent sums of up to 6 paths per pair with their Doppler shifts over
    the frames (10 Hz), a share of the pairs without any path."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    P, F, K = case["pairs"], case["frames"], 6
    r = lambda *s: torch.rand(s, generator=gen, device="cuda", dtype=torch.float64)
    amp = 1e-5 * r(P, K) * (r(P, K) < 0.7)
    amp[:, :2] = 1e-5 * (0.3 + r(P, 2))
    amp = amp * (r(P, 1) < 0.8)
    fd, ph = 117.0 * (2 * r(P, K) - 1), r(P, K)
    h = torch.empty((F, P, 2), dtype=torch.float64, device="cuda")
    for t in range(F):
        a = 2 * math.pi * torch.frac(fd * (0.1 * t) + ph)
        h[t, :, 0] = (amp * torch.cos(a)).sum(1)
        h[t, :, 1] = (amp * torch.sin(a)).sum(1)
    return h


# ---------------------------------------------------------------------------
# one pass
def _loss(S, h):
    p = S["power"] * (h ** 2).sum(-1).sum(0)
    m = S["mask"]
    dbm = 10 * torch.log10(torch.where(m, p, torch.ones_like(p)) * 1e3)
    return (torch.where(m, dbm - S["target"], torch.zeros_like(p)) ** 2).sum()


def run(S):
    op = S["case"]["op"]
    if op == "correlation":
        return [engine.channel_correlation(S["h"], S["lag"])]
    if op == "batch":
        for g, f in zip(S["scenes"], S["frames"]):
            g.update(f)
        S["batch"].trace_async()
        return [[o.rec, o.count] for o in S["batch"].outs]
    g = S["scene"]
    if op == "host_frame":
        g.update(S["frame"])
        out = S["out"]
        g.trace_async(out)
        ch = g.channel(out, S["freq"], out=S["chs"][0])
        g.sync()
        return [out.rec, out.count, ch.path, ch.pair, ch.rx.cpu().numpy()]
    if op == "frame":
        g.update(S["frame"])
        g.trace_async(S["out"], static_cache=S["static"])
        chs = g.channels(S["out"], S["freqs"], outs=S["chs"])
        return [S["out"].rec, S["out"].count, _stack(chs)]
    if op == "cached":
        # from the path cache kept of the frame before
        cache = S["cache"]
        cache.rec.copy_(S["kept"].rec)
        cache.count.copy_(S["kept"].count)
        g.update(S["frame"])
        g.rediscover(cache, n_rays=S["n_low"], static_cache=S["static"], revalidate=True)
        chs = g.channels(cache, S["freqs"], outs=S["chs"])
        return [cache.rec, cache.count, _stack(chs)]
    if op == "fields":
        return _stack(g.channels(S["paths"], S["freqs"], outs=S["chs"]))
    if op == "gradient":
        h = autograd.field(S["eps"], S["sig"], S["tx"], g, S["paths"], S["freq"])
        loss = _loss(S, h)
        return [h.detach(), loss.detach(),
                torch.autograd.grad(loss, (S["eps"], S["sig"], S["tx"]))]
    if op == "revalidate":
        cache = S["cache"]
        cache.rec.copy_(S["paths"].rec)
        cache.count.copy_(S["paths"].count)
        if S["keep"]:
            g.revalidate(cache, keep=True)
            return [cache.rec, cache.count]
        return [g.revalidate_cache(cache), cache.rec, cache.count]
    if op == "backward":
        g.trace_backward_async(S["out"], S["ids"], n_rays=S["case"]["n_rays"])
        return [S["out"].rec, S["out"].count]
    if op == "schedule":
        g.update(S["frame"])
        s = S["sched"]
        g.refresh_schedule(s)
        return [s.state, s.los_ref, s.ids, s.n_due]
    raise ValueError(op)


# ---------------------------------------------------------------------------
# what a pass cannot do without: inputs read and outputs written once; per ray
# one descent of a binary tree over the triangles (a slab test a level) and
# one ray/triangle test; per path its field from the image method
_SLAB, _TRI, _FIELD = 18, 60, 800


def _sizes(case):
    if case["scene"] == "toy":
        return 242, 121, 0, 1, 16
    b = 10 if case["scene"] == "district" else case["blocks"]
    tris = b * b * 4 * 46 + 2 * (b if case["scene"] == "city" else 2 * b) ** 2
    return tris, b * b * 4 * 16, case["n_veh"], 2 if case["scene"] == "district" else 4, \
        case["n_rx"]


def work(case):
    op = case["op"]
    if op == "correlation":
        F, P, L = case["frames"], case["pairs"], case["lag"] + 1
        return {"bytes": 16 * F * P + 8 * P * L, "flops": F * P * (4 + 2 * L)}
    if op == "batch":
        w = {"bytes": 0, "flops": 0}
        for d in _batch_descs(case["n"]):
            n_tri, n_tx = len(d.tri_xyz), len(d.lanes["tx_pos"])
            w["bytes"] += 48 * n_tri + 24 * (d.n_vehicles + len(d.lanes["rxv_veh"]))
            w["flops"] += n_tx * d.n_rays * (_SLAB * math.log2(n_tri) + _TRI)
        return w
    T, F, V, X, R = _sizes(case)
    poses = 24 * (V + R + X)
    ray = _SLAB * math.log2(T) + _TRI
    paths = X * R // 4 + 1     # about a quarter of the pairs hold a path
    nf = case.get("freqs", 1)
    fields = (32 + 32 * nf) * paths + nf * (64 * X * R + 16 * R)
    if op in ("host_frame", "frame"):
        return {"bytes": 48 * T + poses + 32 * paths + fields,
                "flops": X * case["n_rays"] * ray + nf * paths * _FIELD}
    if op == "cached":
        return {"bytes": 48 * T + poses + 64 * paths + fields,
                "flops": X * (case["n_rays"] // 10) * ray + nf * paths * _FIELD}
    if op == "fields":
        return {"bytes": 32 * F + poses + fields, "flops": nf * paths * _FIELD}
    if op == "gradient":
        return {"bytes": 32 * F + poses + 64 * paths + 32 * X * R, "flops": 4 * paths * _FIELD}
    if op == "revalidate":
        return {"bytes": 48 * T + poses + 64 * paths, "flops": 2 * paths * ray}
    if op == "backward":
        n = case["n_ids"]
        return {"bytes": 48 * T + poses + 32 * n * X, "flops": n * case["n_rays"] * ray}
    return {"bytes": 48 * T + poses + 17 * R + X * R, "flops": X * R * ray}  # schedule


# ---------------------------------------------------------------------------
# the field of a path set and Eq. 1 in 64 bits, plain torch
_C, _EPS0 = 299792458.0, 8.8541878128e-12


def _planes(desc, frame, rec):
    """Unit normal, offset, material and velocity of every reflection."""
    off, xyz = desc.face_off.astype(np.int64), desc.face_xyz.astype(np.float64)
    n_faces = desc.n_static_faces
    nxt = np.arange(len(xyz)) + 1
    nxt[off[1:] - 1] = off[:-1]
    a, b = xyz, xyz[nxt]
    newell = np.stack([(a[:, 1] - b[:, 1]) * (a[:, 2] + b[:, 2]),
                       (a[:, 2] - b[:, 2]) * (a[:, 0] + b[:, 0]),
                       (a[:, 0] - b[:, 0]) * (a[:, 1] + b[:, 1])], 1)
    n = np.add.reduceat(newell, off[:-1])
    n /= np.linalg.norm(n, axis=1, keepdims=True)
    centre = np.add.reduceat(xyz, off[:-1]) / np.diff(off)[:, None]
    d = (n * centre).sum(1)
    pos, half = frame.veh_pos.cpu().numpy(), desc.veh_half
    lo, hi = (pos - half).astype(np.float64), (pos + half).astype(np.float64)
    vn, vd = np.zeros((len(pos), 6, 3)), np.zeros((len(pos), 6))
    for j in range(6):
        vn[:, j, j >> 1] = 1.0 if j & 1 else -1.0
        vd[:, j] = hi[:, j >> 1] if j & 1 else -lo[:, j >> 1]
    n, d = np.concatenate([n, vn.reshape(-1, 3)]), np.concatenate([d, vd.reshape(-1)])
    mat = np.concatenate([desc.face_mat.astype(np.int64),
                          np.full(6 * len(pos), desc.veh_mat, np.int64)])
    vel = np.concatenate([np.zeros((n_faces, 3)),
                          np.repeat(frame.veh_vel.cpu().numpy().astype(np.float64), 6, 0)])
    f = np.where(rec[:, 3:7] < len(n), rec[:, 3:7], 0).astype(np.int64)
    dev = functools.partial(torch.as_tensor, device="cuda")
    return dev(n[f]), dev(d[f]), dev(mat[f]), dev(vel[f])


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _vertical(k):
    z = torch.zeros_like(k)
    z[:, 2] = 1.0
    return _unit(z - k[:, 2:3] * k)


def _field64(N, D, mat, vel, depth, tx, rx, vtx, vrx, eps, sig, freqs):
    """(per frequency: complex amplitude), delay and dL/dt of paths of one
    depth; tx, eps and sig may require gradients."""
    img = [tx]
    for q in range(depth):
        img.append(img[q] - N[:, q] * (2 * ((N[:, q] * img[q]).sum(1) - D[:, q]))[:, None])
    pts = [rx]
    for q in range(depth, 0, -1):
        v = pts[0] - img[q]
        t = (D[:, q - 1] - (N[:, q - 1] * img[q]).sum(1)) / (N[:, q - 1] * v).sum(1)
        pts.insert(0, img[q] + v * t[:, None])
    pts.insert(0, tx)
    legs = [pts[q + 1] - pts[q] for q in range(depth + 1)]
    length = sum(v.norm(dim=1) for v in legs)
    k = [_unit(v) for v in legs]
    rate = (vrx * k[-1]).sum(1) - (vtx * k[0]).sum(1)
    for q in range(depth):
        rate = rate + (vel[:, q] * (k[q] - k[q + 1])).sum(1)
    amps = []
    for f in freqs:
        E = _vertical(k[0]).to(torch.complex128)
        for q in range(depth):
            n, kin, kout = N[:, q], k[q], k[q + 1]
            c = (kin * n).sum(1).abs()
            s = _unit(torch.linalg.cross(kin, n))
            ec = torch.complex(eps[mat[:, q]], -sig[mat[:, q]] / (2 * math.pi * f * _EPS0))
            root = torch.sqrt(ec - (1 - c * c))
            gs, gp = (c - root) / (c + root), (ec * c - root) / (ec * c + root)
            es = gs * (E * s).sum(1)
            ep = gp * (E * torch.linalg.cross(s, kin)).sum(1)
            E = es[:, None] * s + ep[:, None] * torch.linalg.cross(s, kout)
        r = (E * _vertical(k[-1])).sum(1)
        lam = _C / f
        ph = -2 * math.pi * (length / lam - torch.floor(length / lam).detach())
        amps.append(r * torch.complex(torch.cos(ph), torch.sin(ph)) * (lam / (4 * math.pi * length)))
    return amps, length / _C, rate


def _paths64(S, eps, sig, tx_pos, freqs):
    """Per frequency [n, 4] (Re a, Im a, tau, f_D) and the pair index of every
    record of the path set S["paths"]."""
    rec = S["paths"].records().astype(np.int64)
    fr = S["frame"]
    N, D, mat, vel = _planes(S["scene"].desc, fr, rec)
    r = torch.as_tensor(rec, device="cuda")
    t, x, depth = r[:, 0], r[:, 1], r[:, 2] & 15
    outs, where = [[] for _ in freqs], []
    for k in range(5):
        i = (depth == k).nonzero()[:, 0]
        if not len(i):
            continue
        amps, tau, rate = _field64(N[i], D[i], mat[i], vel[i], k, tx_pos[t[i]],
                                   fr.rx_pos.double()[x[i]], fr.tx_vel.double()[t[i]],
                                   fr.rx_vel.double()[x[i]], eps, sig, freqs)
        where.append(i)
        for o, a, f in zip(outs, amps, freqs):
            o.append(torch.stack([a.real, a.imag, tau, -(f / _C) * rate], 1))
    order = torch.cat(where).argsort()
    return [torch.cat(o)[order] for o in outs], t * len(fr.rx_pos) + x


def _pairs64(path, pair, n_pairs):
    w = path[:, 0] ** 2 + path[:, 1] ** 2
    one = torch.ones_like(w)
    cols = torch.stack([path[:, 0], path[:, 1], w, w * path[:, 3], w * path[:, 2], one], 1)
    s = torch.zeros((n_pairs, 6), dtype=torch.float64, device="cuda").index_add(0, pair, cols)
    p = torch.where(s[:, 2] > 0, s[:, 2], torch.ones_like(s[:, 2]))
    fm, tm = s[:, 3] / p, s[:, 4] / p
    dev = torch.stack([w * (path[:, 3] - fm[pair]) ** 2, w * (path[:, 2] - tm[pair]) ** 2], 1)
    v = torch.zeros((n_pairs, 2), dtype=torch.float64, device="cuda").index_add(0, pair, dev)
    v = v / p[:, None]
    return torch.stack([s[:, 0], s[:, 1], s[:, 2], fm, v[:, 0].sqrt(), tm, v[:, 1].sqrt(),
                        s[:, 5]], 1)


def exact(case, seed):
    op = case["op"]
    if op == "correlation":
        g = _series(case, seed).square().sum(-1).sqrt()
        F = g.shape[0]
        mu = g.mean(0)
        var = ((g - mu) ** 2).mean(0)
        R = [torch.where(var > 0, ((g[:F - t] * g[t:]).mean(0) - mu * mu)
                         / torch.where(var > 0, var, torch.ones_like(var)),
                         torch.zeros_like(var)) if t < F else torch.zeros_like(var)
             for t in range(case["lag"] + 1)]
        return [torch.stack(R, 1)]
    if op not in ("fields", "gradient"):
        return None  # whole numbers, or a discovery that plain code needs hours for
    S = prepare(case, seed)
    g, d = S["scene"], S["scene"].desc
    tx = S["frame"].tx_pos.double()
    if op == "fields":
        out = []
        paths, pair = _paths64(S, g.eps_r, g.sigma, tx, S["freqs"])
        for p in paths:
            whole = torch.zeros((S["paths"].capacity, 4), dtype=torch.float64, device="cuda")
            whole[:len(p)] = p
            st = _pairs64(p, pair, g.n_tx * g.n_rx).reshape(g.n_tx, g.n_rx, 8)
            # the spreads are differences of nearly equal sums: no value at the
            # accuracy of the other columns
            coh, inc = (st[..., :2] ** 2).sum(-1).sum(0), st[..., 2].sum(0)
            out.append([whole, None, d.tx_power_w * torch.stack([coh, inc], 1)])
        return out
    eps, sig, txp = (S[k].detach().clone().requires_grad_() for k in ("eps", "sig", "tx"))
    (p,), pair = _paths64(S, eps, sig, txp, [S["freq"]])
    h = torch.zeros((g.n_tx * g.n_rx, 2), dtype=torch.float64, device="cuda")
    h = h.index_add(0, pair, p[:, :2]).reshape(g.n_tx, g.n_rx, 2)
    loss = _loss(S, h)
    return [h.detach(), loss.detach(), torch.autograd.grad(loss, (eps, sig, txp))]
