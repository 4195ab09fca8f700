"""What this framework is measured on: the calls its users make, over the sizes they make them.

A case is one pass of a program that keeps a scene, its receivers and a path container and
calls the public entry points (``api.Context``, ``autograd.unfold``).  Kinds of pass:

- ``link``: ``launch`` (ray generation, trace with reception, double-count removal), a
  refinement, ``query``; the paths go into a table of a fixed number of rows in (Tx, Rx, order,
  ray) order, since the library leaves their order open.  With ``move`` the receivers are
  uploaded anew in every pass.
- ``shard``: one rank's ray range of a launch that several GPUs share, its reception records.
- ``merge``: a rank's work after the records were gathered: double-count removal for the pairs
  it owns, refinement, ``query``.
- ``converge``: given paths refined to the double floor (the paper's Figs. 8-9 run 60 iterations).
- ``gradient``: the unfolding of fixed face sequences and its adjoint through autograd.

Meshes come from ``scenes.py``; transmitter and receiver positions, face permittivities and the
gradient inputs come from the seed.  Large meshes are built once per process.
"""
import functools
import math
import weakref

import numpy as np
import torch

from paper_2208_10009_gb300 import _binding as B
from paper_2208_10009_gb300 import api, scenes, shard
from paper_2208_10009_gb300.autograd import unfold

SQ3 = float(np.sqrt(3.0))
TARGET = float(np.radians(0.01))     # the paper's accuracy requirement (AOD and AOA)
C0 = 299792458.0
FREQ = 2.4e9                         # the carrier the refinement defaults to
MANY = 4096                          # a larger table of paths stays on the device


def listed():
    return [
        # a single link in a 10 x 8 x 3 m room: the smallest whole call, launches and latency
        dict(name="room", kind="link", scene="shoebox", size=1, ntx=1, nrx=1, n=64, order=3, iters=8, K=9,
             target=TARGET, lanes=0, form="batch", launcher=0, diffraction=False, move=False),
        # a cluttered room with no face on a coordinate plane, the equidistant launcher and the
        # one-launch refinement with the paper's six sub-rays, an odd division level
        dict(name="clutter", kind="link", scene="clutter", size=20, ntx=1, nrx=4, n=151, order=3, iters=8, K=6,
             target=0.0, lanes=0, form="plain", launcher=8, diffraction=False, move=False),
        # the urban canyon workload: 10k triangles, 256 receivers, 4.9M rays
        dict(name="canyon", kind="link", scene="canyon", size=20, ntx=1, nrx=256, n=700, order=6, iters=6, K=9,
             target=0.0, lanes=32, form="batch", launcher=0, diffraction=False, move=False),
        # the same with order-1 diffraction on the buildings' edges
        dict(name="canyon_diffraction", kind="link", scene="canyon", size=20, ntx=1, nrx=256, n=700, order=6, iters=6,
             K=9, target=0.0, lanes=32, form="batch", launcher=0, diffraction=True, move=False),
        # receivers that move along the canyon's streets: uploaded in every pass
        dict(name="street_walk", kind="link", scene="canyon", size=20, ntx=1, nrx=4096, n=300, order=6, iters=6, K=9,
             target=0.0, lanes=0, form="batch", launcher=0, diffraction=False, move=True),
        # the office workload at 4 transmitters: about a million paths, refinement dominates
        dict(name="office", kind="link", scene="office", size=400, ntx=4, nrx=1024, n=128, order=6, iters=8, K=16,
             target=TARGET, lanes=1, form="batch", launcher=0, diffraction=False, move=False),
        # the large city workload: 1.07M triangles, 4 x 4096 pairs, 194M rays, FP64 tail
        dict(name="city", kind="link", scene="city", size=60, ntx=4, nrx=4096, n=2200, order=8, iters=16, K=9,
             target=0.0, lanes=1, form="batch", launcher=0, diffraction=False, move=False),
        # one rank of four of the same launch: its ray range and its reception records
        dict(name="city_shard", kind="shard", scene="city", size=60, ntx=4, nrx=4096, n=2200, order=8, rank=2, world=4),
        # rank 1 of 2 of the office after the records were gathered
        dict(name="office_merge", kind="merge", scene="office", size=400, ntx=4, nrx=1024, n=128, order=6, iters=8,
             K=16, target=TARGET, lanes=1, rank=1, world=2),
        # convergence to the double floor of every path of 64 room links, lossy walls
        dict(name="converge", kind="converge", nrx=64, order=3, n=64, iters=60, K=6),
        # gradients of a batch of paths in an optimisation loop, and of all paths of the office map
        dict(name="gradient_batch", kind="gradient", paths=4099, order=6),
        dict(name="gradient_map", kind="gradient", paths=3_730_001, order=6),
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["link", "link", "link", "shard", "merge", "converge", "gradient", "gradient"])
    if kind == "converge":
        return dict(kind=kind, nrx=_log(rng, 1, 160), order=rng.randint(1, 3), n=rng.randint(32, 200),
                    iters=rng.randint(20, 60), K=rng.choice([6, 7, 9]))
    if kind == "gradient":
        return dict(kind=kind, paths=_log(rng, 64, 3_700_000), order=rng.randint(1, 8))
    scene = "office" if kind == "merge" else "city" if kind == "shard" else \
        rng.choice(["shoebox", "clutter", "canyon", "canyon", "office", "city"])
    c = dict(kind=kind, scene=scene)
    if scene == "shoebox":
        c |= dict(size=1, ntx=rng.randint(1, 4), nrx=_log(rng, 1, 64), n=_log(rng, 24, 300), order=rng.randint(1, 5))
    elif scene == "clutter":
        c |= dict(size=rng.randint(6, 40), ntx=1, nrx=_log(rng, 1, 40), n=_log(rng, 32, 400), order=rng.randint(1, 4))
    elif scene == "canyon":
        c |= dict(size=rng.randint(18, 20), ntx=rng.randint(1, 2), nrx=_log(rng, 16, 4096), n=_log(rng, 100, 800),
                  order=rng.randint(2, 8))
    elif scene == "office":
        c |= dict(size=rng.randint(60, 400), ntx=rng.randint(1, 4), nrx=_log(rng, 64, 1024), n=_log(rng, 48, 128),
                  order=rng.randint(2, 6))
    else:
        c |= dict(size=rng.randint(12, 60), ntx=rng.randint(1, 4), nrx=rng.randint(12, 64) ** 2,
                  n=_log(rng, 500, 2200), order=rng.randint(3, 8))
    if kind == "shard":
        world = rng.choice([2, 4, 8])
        return c | dict(rank=rng.randrange(world), world=world)
    early = scene in ("shoebox", "office") or rng.random() < 0.3
    c |= dict(iters=rng.randint(5, 16), K=rng.choice([6, 7, 9, 16]), target=TARGET if early else 0.0,
              lanes=1 if scene in ("office", "city") else rng.choice([0, 0, 8, 16, 32]))
    if kind == "merge":
        world = rng.choice([2, 4])
        return c | dict(rank=rng.randrange(world), world=world)
    return c | dict(form=rng.choice(["batch", "batch", "batch", "plain"]) if scene != "office" else "batch",
                    launcher=rng.choice([0, 0, 0, 8, 20]), diffraction=scene == "canyon" and rng.random() < 0.3,
                    move=rng.random() < 0.2)


# ------------------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=3)
def _large(name, size, ntx, nrx):
    if name == "city":
        return scenes.large_city(blocks=size, terrain_cells=round(700 * size / 60), ntx=ntx, nrx=nrx)
    return scenes.office(nbox=size, ntx=ntx, nrx=nrx)


def _geometry(case, seed):
    """Scene, transmitters and receivers of a link, shard or merge case."""
    rng = np.random.default_rng([seed, 11])
    name, size, ntx, nrx = case["scene"], case["size"], case["ntx"], case["nrx"]
    if name == "shoebox":
        sc = scenes.shoebox()
        box = np.array([10.0, 8.0, 3.0])
        return sc, scenes.f32_exact(rng.uniform(0.3, box - 0.3, (ntx, 3))), \
            scenes.f32_exact(rng.uniform(0.3, box - 0.3, (nrx, 3)))
    if name == "clutter":
        return scenes.random_clutter(seed=int(rng.integers(1 << 30)), nbox=size, nrx=nrx)
    if name == "canyon":
        sc, _, _ = scenes.urban_canyon(seed=int(rng.integers(1 << 30)), blocks=size)
        line = 47.5 + 55.0 * np.arange(size - 1)            # street centre lines
        mid = line[size // 4:size - 1 - size // 4]
        tx = np.stack([rng.choice(mid, ntx), rng.choice(mid, ntx), rng.uniform(8, 30, ntx)], -1)
        a, b = rng.choice(line[1:-1], nrx), rng.uniform(40.0, 55.0 * size - 40.0, nrx)
        flip = rng.random(nrx) < 0.5
        rx = np.stack([np.where(flip, b, a), np.where(flip, a, b), rng.uniform(1.5, 20.0, nrx)], -1)
        return sc, scenes.jitter(rng, tx, 1.0), scenes.jitter(rng, rx, 1.0)
    sc, tx, rx = _large(name, size, ntx, nrx)
    by = 0.04 if name == "office" else 0.5                  # stays in free space
    return sc, scenes.jitter(rng, tx, by), scenes.jitter(rng, rx, by)


@functools.lru_cache(maxsize=1)
def _context():
    return api.Context(0)


class State:
    """What a program keeps between passes; its handles close with it."""

    def hold(self, *handles):
        for h in handles:
            weakref.finalize(self, h.close)


def _room_count(order):
    """Specular paths of a rectangular room up to the order: 4 k^2 + 2 of order k and the direct one."""
    return 1 + sum(4 * k * k + 2 for k in range(1, order + 1))


def _pow2(x):
    return 1 << max(6, math.ceil(math.log2(x)))


def _rows(case):
    """Rows of the table that a program keeps for its paths (a shard: for its records)."""
    pairs = case.get("ntx", 1) * case["nrx"]
    if case["kind"] == "converge":
        return pairs * _room_count(case["order"])
    if case["kind"] == "shard":
        return _pow2(pairs * 8)
    per_pair = {"shoebox": 1.5 * _room_count(case["order"]), "clutter": 20 + 10 * case["order"] ** 2,
                "canyon": 32 if case.get("diffraction") else 16, "office": 256, "city": 4}[case["scene"]]
    return _pow2(pairs * per_pair / (case["world"] if case["kind"] == "merge" else 1))


def _container(ctx, s, case):
    """A container sized by one synchronous launch, grown while it overflows (what a program
    does once per scene)."""
    cap_r, cap_p = 1 << 21, 1 << 20
    while True:
        p = ctx.paths_create(cap_r, cap_p)
        try:
            ctx.launch(s.scene, s.tx, s.rxs, p, case["n"], case["order"], rx_angle_scale=SQ3, sync=True, **s.opts)
            st = ctx.launch_stats(p)
            break
        except api.SbrError as e:
            if e.status != 5:
                raise
            st = ctx.launch_stats(p)
            cap_r = max(cap_r, 2 * st["records"], int(st["diffraction_candidates"] / 1.25) + 1)
            cap_p = max(cap_p, 2 * st["paths"])
        finally:
            p.close()
    rec = max(2 * st["records"], int(st["diffraction_candidates"] / 1.25) + 1, 1024)
    return ctx.paths_create(rec, max(2 * st["paths"], 256)), st


def prepare(case, seed):
    ctx = _context()
    s = State()
    s.ctx, s.case = ctx, case
    if case["kind"] == "gradient":
        return _prepare_gradient(s, case, seed)
    if case["kind"] == "converge":
        return _prepare_converge(s, case, seed)
    sc, tx, rx = _geometry(case, seed)
    s.scene = ctx.scene_from(sc)
    s.rxs = ctx.rx_upload(rx)
    s.rx_host = np.asarray(rx, np.float32)
    s.tx = torch.as_tensor(np.asarray(tx, np.float32), device="cuda")
    s.opts = {}
    if case["kind"] == "link":
        s.opts = dict(launcher=case["launcher"], diffraction=case["diffraction"])
    s.paths, st = _container(ctx, s, case)
    s.hold(s.scene, s.rxs, s.paths)
    if case["kind"] == "shard":
        s.rows = max(_rows(case), _pow2(st["records"]) if st["records"] > _rows(case) else 0)
        s.range = shard.ray_range(B.load().sbr_num_rays(case["n"]), case["rank"], case["world"])
        s.buf = torch.empty(s.paths.record_cap * 64, dtype=torch.uint8, device="cuda")
        return s
    if case["kind"] == "merge":   # the gathered records of all ranks
        ctx.launch(s.scene, s.tx, s.rxs, s.paths, case["n"], case["order"], rx_angle_scale=SQ3, records_only=True)
        buf = torch.empty(s.paths.record_cap * 64, dtype=torch.uint8, device="cuda")
        buf, count = ctx.records(s.paths, buf)
        s.gathered = _sorted_records(buf, count, case["nrx"], count).view(torch.uint8).reshape(-1)
    s.rows = max(_rows(case), _pow2(st["paths"]) if st["paths"] > _rows(case) else 0)
    s.out = torch.empty(s.paths.path_cap * 128, dtype=torch.uint8, device="cuda") if s.rows > MANY else None
    return s


def _table(rows, key, size):
    """The rows in the order of their keys, zeros up to the table's size."""
    table = rows.new_zeros((size, rows.shape[1]))
    torch.index_select(rows, 0, torch.argsort(key), out=table[:len(rows)])
    return table


def _sorted_records(buf, count, nrx, size):
    """Reception records (64 bytes each) in (tx, rx, order, ray) order."""
    rows = buf[: count * 64].view(torch.int64).view(-1, 8)
    i = rows.view(torch.int32)
    key = ((i[:, 0].long() * nrx + i[:, 1]) << 40) + (i[:, 3].long() << 32) + i[:, 2]
    return _table(rows, key, size)


# ------------------------------------------------------------------------------- passes
def run(s):
    return _RUN[s.case["kind"]](s)


def _run_link(s):
    c, ctx = s.case, s.ctx
    rxs = ctx.rx_upload(s.rx_host) if c["move"] else s.rxs
    ctx.launch(s.scene, s.tx, rxs, s.paths, c["n"], c["order"], rx_angle_scale=SQ3, **s.opts)
    if c["form"] == "plain":
        ctx.refine(s.scene, s.paths, c["iters"], c["K"], target=c["target"])
    else:
        ctx.batch_refine(s.scene, s.paths, c["iters"], c["K"], target=c["target"], lanes_per_path=c["lanes"])
    out = _query(s)
    if c["move"]:
        rxs.close()
    return out


def _run_shard(s):
    c, ctx = s.case, s.ctx
    ctx.launch(s.scene, s.tx, s.rxs, s.paths, c["n"], c["order"], rx_angle_scale=SQ3, ray_range=s.range,
               records_only=True)
    buf, count = ctx.records(s.paths, s.buf)
    rows = _sorted_records(buf, count, c["nrx"], s.rows)
    i, f = rows.view(torch.int32), rows.view(torch.float32)
    return {"keys": i[:, :12], "measures": f[:, 12:14]}


def _run_merge(s):
    c, ctx = s.case, s.ctx
    ctx.records_dedup(s.paths, s.gathered, rank=c["rank"], world=c["world"])
    ctx.batch_refine(s.scene, s.paths, c["iters"], c["K"], target=c["target"], lanes_per_path=c["lanes"])
    return _query(s)


def _query(s):
    """The refined paths in (tx, rx, order, ray, first face) order; a ray diffracts on several
    wedges, so its first face tells its order-1 paths apart."""
    nrx = s.case["nrx"]
    if s.out is None:
        r = s.ctx.query(s.paths)
        key = ((r["tx"].astype(np.int64) * nrx + r["rx"]) << 49) + (r["order"].astype(np.int64) << 45) + \
            (r["ray"].astype(np.int64) << 14) + (r["faces"][:, 0] & 0x3FFF)
        table = np.zeros(s.rows, B.PATH_DTYPE)
        np.take(r, np.argsort(key), out=table[:len(r)])
        return _fields(torch.from_numpy(table.view(np.int64).reshape(-1, 16)))
    buf, count = s.ctx.query(s.paths, s.out)
    rows = buf[: count * 128].view(torch.int64).view(-1, 16)
    i = rows.view(torch.int32)
    key = ((i[:, 0].long() * nrx + i[:, 1]) << 49) + (i[:, 3].long() << 45) + (i[:, 2].long() << 14) + \
        (i[:, 4] & 0x3FFF)
    return _fields(_table(rows, key, s.rows))


def _fields(rows):
    """The columns of 128-byte path records by their type."""
    i, f, d = rows.view(torch.int32), rows.view(torch.float32), rows.view(torch.float64)
    return {"keys": i[:, :12], "rough": f[:, 12:14], "result": i[:, 14:16], "dir": d[:, 8:11], "err": d[:, 11],
            "delay": d[:, 12], "aod": f[:, 26:28], "aoa": f[:, 28:30], "power": f[:, 30], "flags": i[:, 31]}


# ------------------------------------------------------------------------- convergence
def _room_paths(case, seed):
    """Every specular path of the room up to the order by the image method (FP64): one row per
    path with its receiver, faces, directions, length and the product of its reflection losses."""
    rng = np.random.default_rng([seed, 12])
    box = np.array([10.0, 8.0, 3.0])
    tx = scenes.f32_exact(rng.uniform(0.3, box - 0.3, (1, 3)))
    rx = scenes.f32_exact(rng.uniform(0.3, box - 0.3, (case["nrx"], 3)))
    eps = scenes.f32_exact(rng.uniform(3.0, 7.0, 6))
    axis, at = np.repeat(np.arange(3), 2), np.stack([np.zeros(3), box], -1).reshape(-1)
    seqs = [()]
    for k in range(case["order"]):
        seqs += [q + (f,) for q in seqs if len(q) == k for f in range(6) if not q or q[-1] != f]
    rows = []
    for q in seqs:
        image = rx.copy()                                   # Rx seen from Tx through the faces
        for f in q[::-1]:
            image[:, axis[f]] = 2 * at[f] - image[:, axis[f]]
        w = image - tx
        length = np.linalg.norm(w, axis=1)
        d0 = w / length[:, None]
        o, d, ok, loss = np.repeat(tx, len(rx), 0), d0.copy(), np.ones(len(rx), bool), np.zeros(len(rx))
        for f in q:
            a = axis[f]
            with np.errstate(all="ignore"):
                t = (at[f] - o[:, a]) / d[:, a]
            o = o + np.where(np.isfinite(t), t, 0.0)[:, None] * d
            o[:, a] = at[f]
            ok &= np.isfinite(t) & (t > 1e-3) & np.all((o > 1e-3) | (np.arange(3) == a), 1) & \
                np.all((o < box - 1e-3) | (np.arange(3) == a), 1)
            ci = np.abs(d[:, a])
            r = np.sqrt(eps[f] - (1.0 - ci * ci))
            loss += 20.0 * np.log10(np.abs((ci - r) / (ci + r)))
            d[:, a] = -d[:, a]
        ok &= np.sum((rx - o) * d, 1) > 1e-3
        v = (o if q else np.repeat(tx, len(rx), 0)) - rx
        for i in np.flatnonzero(ok):
            rows.append((i, q, d0[i], length[i], v[i], loss[i]))
    return tx, rx, eps, rows


def _meets(tx, d, faces, order):
    """Whether each direction meets its faces' planes in order."""
    axis, at = np.repeat(np.arange(3), 2), np.array([0.0, 10.0, 0.0, 8.0, 0.0, 3.0])
    d, o, ok, i = d.astype(np.float64), np.repeat(tx, len(d), 0), np.ones(len(d), bool), np.arange(len(d))
    for j in range(int(order.max(initial=0))):
        on, a, h = order > j, axis[faces[:, j]], at[faces[:, j]]
        with np.errstate(all="ignore"):
            t = (h - o[i, a]) / d[i, a]
        ok &= ~on | (np.isfinite(t) & (t > 1e-3))
        o = np.where((on & ok)[:, None], o + np.nan_to_num(t)[:, None] * d, o)
        d[i, a] = np.where(on, -d[i, a], d[i, a])
    return ok


def _prepare_converge(s, case, seed):
    ctx, rng = s.ctx, np.random.default_rng([seed, 13])
    tx, rx, eps, rows = _room_paths(case, seed)
    sc = scenes.shoebox()
    sc.face_eps = eps
    s.scene, s.rxs = ctx.scene_from(sc), ctx.rx_upload(rx)
    theta = api.theta_launch(case["n"])
    r = np.zeros(len(rows), B.PATH_DTYPE)
    d = np.array([x[2] for x in rows])
    off = rng.normal(size=d.shape)
    off -= np.sum(off * d, 1)[:, None] * d
    off /= np.linalg.norm(off, axis=1)[:, None]
    ang = theta * np.sqrt(rng.uniform(0.01, 1.0, len(d)))[:, None]
    r["rx"] = [x[0] for x in rows]
    r["ray"] = np.arange(len(rows))
    r["order"] = [len(x[1]) for x in rows]
    r["faces"] = [x[1] + (-1,) * (8 - len(x[1])) for x in rows]
    for _ in range(8):                                      # a traced ray meets its faces in order
        rough = (d * np.cos(ang) + off * np.sin(ang)).astype(np.float32)
        ang = np.where(_meets(tx, rough, r["faces"], r["order"])[:, None], ang, ang / 2)
    r["dir"] = rough
    r["rough_err"] = r["err"] = ang[:, 0]
    r["rough_dray"] = [x[3] for x in rows]
    s.given, s.tx = r, np.asarray(tx, np.float32)
    s.paths = ctx.paths_create(1024, max(len(r), 1))
    s.hold(s.scene, s.rxs, s.paths)
    s.table = np.zeros(_rows(case), B.PATH_DTYPE)
    return s


def _run_converge(s):
    c, ctx = s.case, s.ctx
    ctx.paths_import(s.paths, s.given, s.tx, s.rxs, c["n"])
    ctx.batch_refine(s.scene, s.paths, c["iters"], c["K"])
    ctx.query(s.paths, s.table)                             # in the order they were given
    return _fields(torch.from_numpy(s.table.view(np.int64).reshape(-1, 16)))


def _exact_converge(case, seed):
    if case["iters"] < 50:
        return None                                         # not at the double floor yet
    _, _, _, rows = _room_paths(case, seed)
    d, v = np.array([x[2] for x in rows]), np.array([x[4] for x in rows])
    length, loss = np.array([x[3] for x in rows]), np.array([x[5] for x in rows])
    table = lambda x: np.concatenate([x, np.zeros((_rows(case) - len(x),) + x.shape[1:])])
    angles = lambda w: np.stack([np.arctan2(w[:, 1], w[:, 0]), np.arctan2(w[:, 2], np.hypot(w[:, 0], w[:, 1]))], -1)
    power = 20.0 * np.log10(C0 / FREQ / (4.0 * np.pi * length)) + loss
    return {"keys": None, "rough": None, "result": None, "dir": table(d), "err": None,
            "delay": table(length / C0), "aod": table(angles(d)), "aoa": table(angles(v)), "power": table(power),
            "flags": None}


# ---------------------------------------------------------------------------- gradients
@functools.lru_cache(maxsize=1)
def _canyon_planes():
    """The default canyon and its faces' planes (n, h) in FP64 (first triangle of each)."""
    sc, _, _ = scenes.urban_canyon()
    first = np.full(sc.nf, -1)
    first[sc.tri_face[::-1]] = np.arange(sc.nt)[::-1]
    a, b, c = (sc.verts[sc.tris[first, k]] for k in range(3))
    n = np.cross(b - a, c - a)
    n /= np.linalg.norm(n, axis=1)[:, None]
    return sc, np.concatenate([n, np.sum(n * a, 1)[:, None]], 1)


def _gradient_inputs(case, seed):
    """Paths of the canyon: a transmitter over a street, a receiver within 150 m, a sequence of
    walls of the blocks around them, roofs and the ground; the launch direction is within the
    cone of the unfolded one (what the refinement leaves)."""
    sc, planes = _canyon_planes()
    g = torch.Generator(device="cuda").manual_seed(seed)
    P, dev = case["paths"], "cuda"
    u = lambda *shape: torch.rand(*shape, generator=g, device=dev, dtype=torch.float64)
    block = (u(P, 2) * 14).long() + 3                       # the transmitter's block
    tx = torch.cat([block * 55.0 + 47.5 + (u(P, 2) - 0.5) * 10, 5 + 25 * u(P, 1)], 1).float()
    rx = torch.cat([tx[:, :2] + (u(P, 2) - 0.5) * 200, 1.5 + 18 * u(P, 1)], 1).float()
    near = (block[:, None, :] + (u(P, 8, 2) * 4).long() - 1)
    faces = 1 + (near[..., 0] * 20 + near[..., 1]) * 5 + (u(P, 8) * 5).long()
    faces = torch.where(u(P, 8) < 0.25, 0, faces)           # the ground
    step = (faces[:, 1:] == faces[:, :-1]) & (faces[:, 1:] > 0)
    faces[:, 1:] -= step.long()                             # no face twice in a row
    order = 1 + (u(P) * case["order"]).long()
    faces = torch.where(torch.arange(8, device=dev) < order[:, None], faces, -1)
    pl = torch.as_tensor(planes, device=dev)
    _, w, _ = _unfold64(pl, tx.double(), rx.double(), None, faces, order)
    az = torch.atan2(w[:, 1], w[:, 0]) + (u(P) - 0.5) * 1e-3
    el = torch.atan2(w[:, 2], torch.hypot(w[:, 0], w[:, 1])) + (u(P) - 0.5) * 1e-3
    grad = torch.randn(P, 8, generator=g, device=dev)
    return sc, pl, tx, rx, torch.stack([az, el], -1).float(), faces.int(), order.int(), grad


def _unfold64(pl, tx, rx, az_el, faces, order):
    """The unfolding in FP64: the outputs (none without az_el), w = Rx' - Tx and v = Tx's last image - Rx."""
    mirror = lambda x, p, on: torch.where(on[:, None], x - 2 * (torch.sum(x * p[:, :3], 1) - p[:, 3])[:, None] * p[:, :3], x)
    plane = [pl[faces[:, j].clamp(min=0).long()] for j in range(8)]
    on = [order > j for j in range(8)]
    x, t = rx, tx
    for j in range(7, -1, -1):
        x = mirror(x, plane[j], on[j])
    for j in range(8):
        t = mirror(t, plane[j], on[j])
    w, v = x - tx, t - rx
    if az_el is None:
        return None, w, v
    ce, se = torch.cos(az_el[:, 1]), torch.sin(az_el[:, 1])
    d = torch.stack([ce * torch.cos(az_el[:, 0]), ce * torch.sin(az_el[:, 0]), se], -1)
    miss = w - torch.sum(w * d, 1)[:, None] * d
    for j in range(8):                                      # back to the real space: A^T
        p = plane[j][:, :3]
        miss = torch.where(on[j][:, None], miss - 2 * torch.sum(miss * p, 1)[:, None] * p, miss)
    angles = lambda y: [torch.atan2(y[:, 1], y[:, 0]), torch.atan2(y[:, 2], torch.sqrt(y[:, 0] ** 2 + y[:, 1] ** 2))]
    delay = torch.sqrt(torch.sum(w * w, 1)) / C0
    return torch.cat([miss, torch.stack([delay] + angles(w) + angles(v), -1)], 1), w, v


def _prepare_gradient(s, case, seed):
    sc, _, tx, rx, ae, s.faces, s.order, s.grad = _gradient_inputs(case, seed)
    s.scene = s.ctx.scene_from(sc)
    s.hold(s.scene)
    s.inputs = [x.requires_grad_() for x in (tx, rx, ae)]
    return s


def _run_gradient(s):
    for x in s.inputs:
        x.grad = None
    out = unfold(s.ctx, s.scene, *s.inputs, s.faces, s.order)
    out.backward(s.grad)
    return [out.detach()] + [x.grad for x in s.inputs]


def _exact_gradient(case, seed):
    _, pl, tx, rx, ae, faces, order, grad = _gradient_inputs(case, seed)
    ins = [x.double().requires_grad_() for x in (tx, rx, ae)]
    out, _, _ = _unfold64(pl, *ins, faces, order)
    out.backward(grad.double())
    return [out.detach()] + [x.grad for x in ins]


_RUN = {"link": _run_link, "shard": _run_shard, "merge": _run_merge, "converge": _run_converge,
        "gradient": _run_gradient}


def exact(case, seed):
    """The convergence cases end at the image method's paths; the gradient cases are plain
    FP64 algebra.  A launch has no plain counterpart within the time (194M rays)."""
    if case["kind"] == "converge":
        return _exact_converge(case, seed)
    return _exact_gradient(case, seed) if case["kind"] == "gradient" else None


# --------------------------------------------------------------------------------- work
def work(case):
    """What a pass cannot do without.  A launch: the mesh, the receivers and 16 bytes of every
    path's record pair read and written; per ray-bounce one descent of the mesh's 4-wide tree
    (48 operations a level), one triangle test (40) and the reflection (20).  A refinement:
    per iteration and sub-ray one dot product a face and the error (7 a face, 15)."""
    if case["kind"] == "gradient":
        return {"bytes": case["paths"] * 232.0, "flops": case["paths"] * (40.0 * case["order"] + 150)}
    if case["kind"] == "converge":
        paths = _rows(case)
        return {"bytes": paths * 256.0, "flops": float(paths * case["iters"] * case["K"] * (7 * case["order"] + 15))}
    tris = {"shoebox": 12, "clutter": 48 + 12 * case["size"], "canyon": 6050 + 10 * case["size"] ** 2,
            "office": 19200 + 90 * case["size"], "city": 297 * case["size"] ** 2}[case["scene"]]
    closed = case["scene"] in ("shoebox", "clutter", "office")
    bounces = case["order"] + 1 if closed else min(case["order"] + 1, 2.4)
    rays = case["ntx"] * (10 * case["n"] ** 2 + 2) / (case.get("world", 1) if case["kind"] == "shard" else 1)
    per_pair = {"shoebox": 40, "clutter": 20, "canyon": 2.5, "office": 230, "city": 1.1}[case["scene"]]
    paths = case["ntx"] * case["nrx"] * per_pair
    levels = max(1.0, math.log(tris, 4))
    if case["kind"] == "merge":
        return {"bytes": paths * (1.6 * 64 + 128 / case["world"]),
                "flops": paths / case["world"] * 3 * case["K"] * (7 * case["order"] + 15)}
    flops = rays * bounces * (48 * levels + 60)
    if case["kind"] == "link":
        flops += paths * 3 * case["K"] * (7 * case["order"] + 15)
    return {"bytes": tris * 48.0 + case["nrx"] * 12 + paths * 128, "flops": float(flops)}
