"""The workloads this library is timed on, each through its public binding.

A case names an operation ("op") and its sizes.  Scenes are the synthetic
cities of paper_2208_10008_gb300/scenes.py (extruded convex footprints on a
flat ground, uniform or clustered centres), drawn here on the GPU so that the
large ones take a fraction of a second; a different seed is another city,
other transmitters and other rays.

  listed()            the cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) what a program holds before the call
  run(state)          one pass through the binding and its outputs
  work(case)          bytes a pass cannot do without
  tolerance(case)     how far another correct implementation may be off
  exact(case, seed)   the outputs in float64 by brute force, where affordable
"""
import math

import numpy as np
import torch

from paper_2208_10008_gb300 import rtbvh, scenes

FIB, ICO = rtbvh.RT_RAYS_FIBONACCI, rtbvh.RT_RAYS_ICOSPHERE
METRO = dict(buildings=300000, size=20000.0, sides=16, clusters=20, tmax=3000.0)
CITY = dict(buildings=10000, size=3000.0, sides=8, clusters=0, tmax=1000.0)
MEDIUM = dict(buildings=1000, size=1000.0, sides=8, clusters=0, tmax=500.0)


def listed():
    return [
        # the smallest call: 4,096 rays on the 64-building city, where launches and latency count
        dict(name="closest tiny", op="closest", buildings=64, size=200.0, sides=4, clusters=0, tmax=1000.0, alpha=1.0,
             rays=4096, launch="fibonacci"),
        # rays without order (diffuse queries, ray sets of a user's own) on a 200k-triangle city, an odd count
        dict(name="closest random", op="closest", **CITY, alpha=0.7, rays=262143, launch="random"),
        # 8.4M direct rays of four transmitters on the 13M-triangle metro, a resident tree
        dict(name="closest metro", op="closest", **METRO, alpha=1.0, rays=4 << 21, launch="fibonacci"),
        # line-of-sight of a million point pairs (coverage prediction)
        dict(name="visibility", op="any", **MEDIUM, alpha=0.7, rays=1000003),
        # a scene that moves: new triangles, a new tree and the benchmark's 655,362 rays
        dict(name="step medium", op="rebuild", **MEDIUM, alpha=0.7, rays=8, launch="icosphere"),
        # the same step for a program whose triangles, rays and hits live in page-locked host memory
        dict(name="step medium host", op="host", **MEDIUM, alpha=0.7, rays=8, launch="icosphere"),
        # a new tree over the 13M-triangle metro and the first transmitter's rays
        dict(name="step metro", op="rebuild", **METRO, alpha=0.7, rays=1 << 20, launch="fibonacci"),
        # a tree per transmitter, pruned to its ray action range, in a 4M-triangle metro
        dict(name="step range", op="range", buildings=100000, size=12000.0, sides=16, clusters=20, tmax=2000.0,
             alpha=0.7, rays=1 << 20, launch="fibonacci"),
        # one transmitter, call by call: launch, trace, reflect, trace the survivors, twice
        dict(name="bounce", op="bounce", **CITY, alpha=0.7, rays=1 << 20, orders=2),
        # 16 transmitters with uneven launches, three reflections, visibility to a 64 x 64 grid: one launch
        dict(name="batch", op="batch", **CITY, alpha=0.7, rays=1 << 21, tx=16, orders=3, grid=64),
        # reception of a launch at a street-level receiver grid, records in order of ray and receiver
        dict(name="receive", op="receive", **MEDIUM, alpha=0.7, rays=1 << 21, grid=64),
        # twelve requests of uneven size on three resident scenes, served side by side, hits to the host
        dict(name="serve", op="serve", buildings=20000, size=4622.1, sides=8, clusters=0, tmax=1000.0, alpha=0.7,
             rays=1 << 20, requests=12),
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    op = rng.choice(["closest", "closest", "any", "rebuild", "rebuild", "host", "range", "bounce", "batch", "receive",
                     "serve"])
    b = _log(rng, 64, 10000 if op in ("host", "bounce", "batch", "receive", "serve") else 200000)
    clustered = b >= 30000 or rng.random() < 0.2
    c = dict(op=op, buildings=b, size=round(1000.0 * math.sqrt(b / (750.0 if clustered else 1000.0)) + 150.0, 1),
             sides=rng.choice([4, 8, 16]), clusters=20 if clustered else 0,
             tmax=float(rng.choice([300, 500, 1000, 3000])), alpha=rng.choice([1.0, 0.7, 0.4]))
    if op in ("closest", "rebuild", "host", "range"):
        c["launch"] = rng.choice(["fibonacci", "icosphere", "random"] if op != "range" else ["fibonacci", "icosphere"])
        c["rays"] = rng.randint(3, 9) if c["launch"] == "icosphere" else _log(rng, 1000, (1 << 22) - 1)
    elif op == "any":
        c["rays"] = _log(rng, 1000, (1 << 21) - 1)
    elif op == "receive":  # a launch fine enough that a ray meets few receiving spheres
        c["rays"], c["tmax"] = _log(rng, 1 << 16, (1 << 21) - 1), min(c["tmax"], 1000.0)
    else:
        c["rays"] = _log(rng, 1000, (1 << 20) - 1)
    if op in ("bounce", "batch"):
        c["orders"] = rng.randint(1, 3)
    if op == "batch":
        c["tx"] = rng.randint(1, 16)
    if op in ("batch", "receive"):
        c["grid"] = rng.randint(8, 64)
    if op == "serve":
        c["requests"] = rng.randint(1, 12)
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(int(seed) % (1 << 62))


def city(case, seed, buildings=None, size=None):
    """float32 [T, 3, 3] on the GPU: closed prisms over random convex footprints
    of 4 .. `sides` corners (8 .. 16 in the metro's recipe), heights lognormal(3, 0.5) m, then
    the two ground triangles; and a transmitter place that no building covers."""
    nb, size = buildings or case["buildings"], size or case["size"]
    g = _gen(seed)
    kw = dict(generator=g, device="cuda", dtype=torch.float64)
    lo = 8 if case["sides"] == 16 else 4
    n = torch.randint(lo, case["sides"] + 1, (nb,), generator=g, device="cuda")
    r = 4.0 + 8.5 * torch.rand(nb, **kw)
    if case["clusters"]:
        cc = 12.5 + (size - 25.0) * torch.rand(case["clusters"], 2, **kw)
        k = torch.randint(0, case["clusters"], (nb,), generator=g, device="cuda")
        c = cc[k] + (size / 25.0) * torch.randn(nb, 2, **kw)
        c = torch.minimum(torch.maximum(c, r[:, None]), size - r[:, None])
    else:
        c = r[:, None] + (size - 2 * r[:, None]) * torch.rand(nb, 2, **kw)
    h = torch.exp(3.0 + 0.5 * torch.randn(nb, **kw))
    # transmitters stand a few metres beside random buildings, where no footprint reaches
    at = torch.randint(0, nb, (64,), generator=g, device="cuda")
    spots = torch.cat([c[at] + 14.0, 10.0 + 30.0 * torch.rand(64, 1, **kw)], 1)
    spots[:, :2].clamp_(1.0, size - 1.0)
    for q in range(64):
        far = c - spots[q, :2]
        d = far.norm(dim=1)
        near = d < r + 0.5
        c = torch.where(near[:, None], spots[q, :2] + far / d.clamp_min(1e-3)[:, None] * (r + 1.0)[:, None], c)
    a = torch.rand(nb, case["sides"], **kw) * (2 * math.pi)
    a = torch.where(torch.arange(case["sides"], device="cuda")[None, :] < n[:, None], a, math.inf).sort(dim=1).values
    parts = []
    for m in range(lo, case["sides"] + 1):
        s = (n == m).nonzero()[:, 0]
        if not len(s):
            continue
        xy = c[s, None, :] + r[s, None, None] * torch.stack([a[s, :m].cos(), a[s, :m].sin()], -1)
        bot = torch.cat([xy, torch.zeros_like(xy[..., :1])], -1)
        top = torch.cat([xy, h[s, None, None].expand(-1, m, 1)], -1)
        nxt_b, nxt_t = bot.roll(-1, 1), top.roll(-1, 1)
        f = torch.arange(1, m - 1, device="cuda")
        parts.append(torch.cat([torch.stack([bot, nxt_b, nxt_t], 2), torch.stack([bot, nxt_t, top], 2),
                                torch.stack([top[:, :1].expand(-1, m - 2, 3), top[:, f], top[:, f + 1]], 2),
                                torch.stack([bot[:, :1].expand(-1, m - 2, 3), bot[:, f + 1], bot[:, f]], 2)],
                               1).reshape(-1, 3, 3).float())
    z = size
    parts.append(torch.tensor([[[0, 0, 0], [z, 0, 0], [z, z, 0]], [[0, 0, 0], [z, z, 0], [0, z, 0]]],
                              dtype=torch.float32, device="cuda"))
    return torch.cat(parts).contiguous(), spots.float().cpu().numpy()


def launch(case, seed, spots, count=None):
    """Rays as a program makes them: the library's launches (several transmitters
    beyond 2^21 rays), or origins over the area with uniform directions."""
    n, tmax = count or case["rays"], case["tmax"]
    if case.get("launch") == "icosphere":
        return rtbvh.rt_gen_rays(ICO, spots[0], n, 0.0, tmax)
    if case.get("launch") == "random":
        g = _gen(seed + 77)
        kw = dict(generator=g, device="cuda", dtype=torch.float64)
        o = torch.rand(n, 3, **kw) * torch.tensor([case["size"], case["size"], 59.0], device="cuda", dtype=torch.float64)
        o[:, 2] += 1.0
        d = torch.randn(n, 3, **kw)
        d = d / d.norm(dim=1, keepdim=True)
        z = torch.zeros(n, 1, device="cuda", dtype=torch.float64)
        return torch.cat([o, z, d, z + tmax], 1).float().contiguous()
    k = max(1, -(-n // (1 << 21)))
    per = [n // k + (1 if t < n % k else 0) for t in range(k)]
    return torch.cat([rtbvh.rt_gen_rays(FIB, spots[t], p, 0.0, tmax) for t, p in enumerate(per)])


def pairs(case, seed):
    """Segments between random points over the area: 10-40 m to 1.5-10 m above ground."""
    g = _gen(seed + 99)
    n = case["rays"]
    a, b = (torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64) for _ in range(2))
    s = case["size"]
    a = a * torch.tensor([s, s, 30.0], device="cuda") + torch.tensor([0, 0, 10.0], device="cuda")
    b = b * torch.tensor([s, s, 8.5], device="cuda") + torch.tensor([0, 0, 1.5], device="cuda")
    z = torch.zeros(n, 1, device="cuda", dtype=torch.float64)
    return torch.cat([a, z, b - a, z + 1.0], 1).float().contiguous()


def tree(case, source):
    return dict(alpha=case["alpha"], dist_norm=1, source=tuple(float(v) for v in source), max_leaf=4, bins=16)


def uneven(case):
    """Ray counts of a batch's transmitters or of a session's requests: log-uniform
    from a 32nd of the largest up to it (the case's own, whatever the seed)."""
    rng = np.random.Generator(np.random.PCG64(case["rays"] + 5))
    k = case.get("tx") or case["requests"]
    n = np.exp(rng.uniform(math.log(max(64, case["rays"] // 32)), math.log(case["rays"]), k)).astype(np.int64)
    n[0] = case["rays"]
    return n, rng


class State:
    pass


def _order(n, reflected, rays):
    """A program's buffers for one reflection order of up to n rays."""
    o = {"hits": torch.zeros((n, 4), device="cuda")}
    if rays:
        o["rays"] = torch.zeros((n, 8), device="cuda")
    if reflected:
        o.update({k: torch.zeros(n, dtype=torch.int32, device="cuda") for k in ("skip", "src")},
                 count=torch.zeros(1, dtype=torch.int32, device="cuda"))
    return o


def prepare(case, seed):
    s = State()
    s.case, op = case, case["op"]
    if op == "serve":
        s.scenes, s.spots = [], []
        for j, nb in enumerate(sorted({max(8, case["buildings"] // 16), max(8, case["buildings"] // 4),
                                       case["buildings"]})):
            size = 1000.0 * math.sqrt(nb / 1000.0) + 150.0
            t, sp = city(case, seed + 31 * j, nb, size)
            sc = rtbvh.rt_scene_upload(t)
            rtbvh.rt_bvh_build(sc, **tree(case, (size / 2, size / 2, 25.0)))
            s.scenes.append(sc)
            s.spots.append(sp)
        torch.cuda.synchronize()
        s.session = rtbvh.Session(1 << 30, 8)
        ids = [s.session.add_scene(sc) for sc in s.scenes]
        n, rng = uneven(case)
        which = rng.integers(0, len(ids), len(n))
        s.requests = [(ids[w], s.spots[w][q], int(n[q]), q % 3) for q, w in enumerate(which)]
        return s
    s.tris, s.spots = city(case, seed)
    mid = (case["size"] / 2, case["size"] / 2, 30.0)
    s.tree = tree(case, mid if op in ("batch", "any") or case.get("launch") == "random" else s.spots[0])
    s.scene = rtbvh.rt_scene_upload(s.tris)
    if op not in ("rebuild", "host", "range"):
        rtbvh.rt_bvh_build(s.scene, **s.tree)
    if op == "any":
        s.rays = pairs(case, seed)
    elif op == "batch":
        s.params, _ = uneven(case)
        s.batch = rtbvh.Batch(s.scene, s.spots[: case["tx"]], s.params, FIB, max_order=case["orders"],
                              tmax=case["tmax"], rx_pos=scenes.receiver_grid(case["size"], case["grid"], 10.0))
        s.orders = [_order(int(s.params.sum()), k > 0, False) for k in range(case["orders"] + 1)]
        s.blocked = torch.zeros(case["tx"] * case["grid"] ** 2, dtype=torch.uint8, device="cuda")
    elif op == "bounce":
        s.orders = [_order(case["rays"], k > 0, True) for k in range(case["orders"] + 1)]
    else:
        s.rays = launch(case, seed, s.spots)
    if op == "range":
        s.tree["range"] = case["tmax"]
    if op == "host":
        s.tris = s.tris.cpu().pin_memory()
        s.rays = s.rays.cpu().pin_memory()
        s.hits = torch.empty((s.rays.shape[0], 4)).pin_memory()
    if op == "receive":
        s.hits = rtbvh.rt_trace_closest(s.scene, s.rays)
        s.delta = math.sqrt(4 * math.pi / s.rays.shape[0])
        s.m = case["grid"] ** 2
        s.records = torch.zeros((case["rays"], 4), dtype=torch.int32, device="cuda")
        s.rx = rtbvh.rt_rxset_create(scenes.receiver_grid(case["size"], case["grid"], 1.5),
                                     case["tmax"] * s.delta / math.sqrt(3.0))
    return s


# ------------------------------------------------------------------ one pass
def _hits(h):
    return {"t": h[:, 0], "tri": rtbvh.hit_ids(h), "uv": h[:, 2:]}


def run(s):
    op, case = s.case["op"], s.case
    if op == "closest":
        return _hits(rtbvh.rt_trace_closest(s.scene, s.rays))
    if op == "any":
        return rtbvh.rt_trace_any(s.scene, s.rays)
    if op in ("rebuild", "range"):
        if op == "rebuild":
            rtbvh.rt_scene_update(s.scene, s.tris)
        rtbvh.rt_bvh_build(s.scene, **s.tree)
        return _hits(rtbvh.rt_trace_closest(s.scene, s.rays))
    if op == "host":
        rtbvh.rt_scene_update(s.scene, s.tris)
        rtbvh.rt_bvh_build(s.scene, **s.tree)
        return _hits(rtbvh.rt_trace_closest_host(s.scene, s.rays, s.hits))
    if op == "bounce":
        # buffers of the program's own, one set per order; rows past an order's count stay as they were
        rays, hits, skip = s.orders[0]["rays"], s.orders[0]["hits"], None
        rtbvh.rt_gen_rays(FIB, s.spots[0], case["rays"], 0.0, case["tmax"], rays=rays)
        rtbvh.rt_trace_closest(s.scene, rays, hits)
        for o in s.orders[1:]:
            rtbvh.rt_reflect(s.scene, rays, hits, o["rays"], o["skip"], o["src"], o["count"])
            m = int(o["count"].item())  # the survivors' number, as a program reads it before it goes on
            rays, skip, hits = o["rays"][:m], o["skip"][:m], o["hits"][:m]
            rtbvh.rt_trace_closest(s.scene, rays, hits, skip=skip)
        return [{"rays": o["rays"], **_hits(o["hits"])} if k == 0 else
                {"rays": o["rays"], "src": o["src"], "count": o["count"], **_hits(o["hits"])}
                for k, o in enumerate(s.orders)]
    if op == "batch":
        s.batch.run()
        for k, o in enumerate(s.orders):  # the batch's buffers hold until its next run: the program keeps a copy
            _, hits, src, n = s.batch.order(k)
            o["hits"][:n] = hits
            if k:
                o["src"][:n] = src
        s.blocked.copy_(s.batch.visibility())
        return [_hits(o["hits"]) if k == 0 else {"src": o["src"], **_hits(o["hits"])}
                for k, o in enumerate(s.orders)] + [s.blocked]
    if op == "receive":
        rec, count = rtbvh.rt_receive(s.rx, s.rays, s.hits, s.delta, case["tmax"], max_records=case["rays"])
        n = min(int(count.item()), case["rays"])
        rec = rec[:n]
        s.records[:n] = rec[torch.argsort(rec[:, 0].long() * s.m + rec[:, 1])]
        return {"ray": s.records[:, 0], "rx": s.records[:, 1], "path": s.records[:, 2:].view(torch.float32),
                "count": count}
    if op == "serve":
        tickets = [s.session.submit(sc, tx, FIB, n, k, case["tmax"]) for sc, tx, n, k in s.requests]
        out = []
        for t in tickets:
            s.session.wait(t)
            h, counts = s.session.release(t)
            out.append([h[:, 0], rtbvh.hit_ids(h), h[:, 2:], counts])
        return out
    raise ValueError(op)


# ------------------------------------------------------------------ what a pass costs at least
def _count(case):
    return 10 * 4 ** case["rays"] + 2 if case.get("launch") == "icosphere" else case["rays"]


def _tris(case):
    return case["buildings"] * (4 * ((8 if case["sides"] == 16 else 4) + case["sides"]) // 2 - 4) + 2


def work(case):
    """Rays (32 B) read, hits (16 B) written, triangles (36 B) read, once each."""
    op, n, t = case["op"], _count(case), 36 * _tris(case)
    if op == "any":
        b = 33 * n + t
    elif op == "bounce":  # rays of every order written, hits and parents written; the launch has no input
        b = t + n * (32 + 16) + case["orders"] * n * (32 + 16 + 8) * 0.5
    elif op == "batch":
        total = float(uneven(case)[0].sum())
        b = t + total * (32 + 16) + case["orders"] * total * (32 + 16 + 8) * 0.4
        b += 33 * case["tx"] * case["grid"] ** 2
    elif op == "receive":
        b = 48 * n + 16 * case["grid"] ** 2
    elif op == "serve":
        b = float(uneven(case)[0].sum()) * 16
    else:
        b = 48 * n + t
    return {"bytes": float(b), "flops": 0.0}


def tolerance(case):
    """Hits are the float64 definition's: ids differ only where the two nearest
    hits lie within 1e-6 of each other; t and (u, v) are float32 evaluations
    of them (a grazing hit of a kilometre-sized facet is the worst)."""
    return {"rel": 4e-6, "max": 1e-3, "differ": 1e-5}


# ------------------------------------------------------------------ float64
def _brute(tris, rays, any_hit=False):
    """Moller-Trumbore of every ray against every triangle in float64, one operation
    at a time: inclusive edges, two-sided, |det| <= 1e-14 |e1||e2||d| misses,
    tmin < t < tmax, lowest id on equal t."""
    T, R = tris.double(), rays.double()

    def dot(a, b):
        return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]

    def cross(a, b):
        return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]

    v0 = [T[None, :, 0, k] for k in range(3)]
    e1 = [T[None, :, 1, k] - v0[k] for k in range(3)]
    e2 = [T[None, :, 2, k] - v0[k] for k in range(3)]
    lim = 1e-14 * (dot(e1, e1).sqrt() * dot(e2, e2).sqrt())
    n, step = R.shape[0], max(1, (1 << 25) // T.shape[0])
    t_out = torch.full((n,), math.inf, dtype=torch.float64, device="cuda")
    id_out = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    uv_out = torch.zeros((n, 2), dtype=torch.float64, device="cuda")
    for i in range(0, n, step):
        r = R[i:i + step]
        d = [r[:, 4 + k, None] for k in range(3)]
        p = cross(d, e2)
        det = dot(e1, p)
        inv = 1.0 / det
        s = [r[:, k, None] - v0[k] for k in range(3)]
        u = dot(s, p) * inv
        q = cross(s, e1)
        v = dot(d, q) * inv
        t = dot(e2, q) * inv
        ok = (det.abs() > lim * dot(d, d).sqrt()) & (u >= 0) & (u <= 1) & (v >= 0) & (u + v <= 1)
        ok &= (t > r[:, 3:4]) & (t < r[:, 7:8])
        t = torch.where(ok, t, math.inf)
        best = t.min(dim=1).values
        first = (t == best[:, None]).to(torch.uint8).argmax(dim=1)
        hit = best < math.inf
        t_out[i:i + step] = best
        id_out[i:i + step] = torch.where(hit, first, -1).int()
        for k, w in enumerate((u, v)):
            uv_out[i:i + step, k] = torch.where(hit, w.gather(1, first[:, None])[:, 0], 0.0)
    if any_hit:
        return (id_out >= 0).to(torch.uint8)
    return {"t": t_out, "tri": id_out, "uv": uv_out}


def exact(case, seed):
    if case["op"] not in ("closest", "any", "rebuild", "host", "range", "receive"):
        return None  # chains of reflections: each order's rays are the float32 results of the last
    if case["op"] != "receive" and _count(case) * _tris(case) > 2.5e10:
        return None
    if case["op"] == "receive":
        s = prepare(case, seed)
        o, d = s.rays[:, 0:3].double(), s.rays[:, 4:7].double()
        tmin, tmax = s.rays[:, 3].double(), s.rays[:, 7].double()
        tend = torch.minimum(s.hits[:, 0].double(), tmax)
        rx = torch.from_numpy(scenes.receiver_grid(case["size"], case["grid"], 1.5)).cuda().double()
        dd = (d * d).sum(1)
        k = s.delta / math.sqrt(3.0)
        rec = []
        for i in range(0, len(o), 8192):
            q = rx[None] - o[i:i + 8192, None]
            ts = torch.einsum("rmk,rk->rm", q, d[i:i + 8192]) / dd[i:i + 8192, None]
            dist = (q - ts[..., None] * d[i:i + 8192, None]).norm(dim=2)
            length = (case["tmax"] - tmax[i:i + 8192, None]) + ts
            ok = (ts >= tmin[i:i + 8192, None]) & (ts < tend[i:i + 8192, None]) & (dist <= length * k)
            r, m = ok.nonzero(as_tuple=True)
            rec.append((r + i, m, length[r, m], dist[r, m]))
        r, m, length, dist = (torch.cat(x) for x in zip(*rec))
        out = torch.zeros((case["rays"], 2), dtype=torch.int32, device="cuda")
        path = torch.zeros((case["rays"], 2), dtype=torch.float64, device="cuda")
        k = min(len(r), case["rays"])
        out[:k], path[:k] = torch.stack([r, m], 1)[:k].int(), torch.stack([length, dist], 1)[:k]
        return {"ray": out[:, 0], "rx": out[:, 1], "path": path, "count": torch.tensor([len(r)], dtype=torch.int32)}
    tris, spots = city(case, seed)
    if case["op"] == "any":
        return _brute(tris, pairs(case, seed), True)
    # (a range build: no triangle beyond the range is met by a ray that ends there)
    return _brute(tris, launch(case, seed, spots))
