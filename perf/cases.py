"""Workloads that stand for what a user of bathygrid has it do.

Every case is one pass through the public entry points of
`paper_2505_22675_gb300`, on seeded synthetic inputs: multibeam surveys (256
beams per ping over a +-60 degree fan, pings every half metre, +-1 m position
jitter), uniform tiles, gridded products with missing nodes. Depths are
metres positive down around 3500 m, with relief of tens of metres, 0.5 m
noise and a few rejected beams (NaN). A survey program grids each new set of
soundings once, so the upload and the hash build belong to the pass.
"""
from __future__ import annotations

import math
import weakref

import numpy as np
import torch

import paper_2505_22675_gb300 as bg

SIDES = (64, 128, 256, 512, 1024)   # tile grids of the batched and serving mixes
CELLS_M = (1, 2, 3, 4)
BEAMS = 256
ALTITUDE_M = 100.0
FAN_DEG = 60.0
PING_STEP_M = 0.5
LINE_SPACING_M = 500.0


def listed():
    return [
        # the smallest tile of a survey mix: latency and launches decide
        dict(name="tile_small_idw", kind="grid", survey="uniform", n=1_000, side_cm=6_400,
             cell_cm=100, nx=64, ny=64, method="idw", k=16, power=2.0, nbr=False),
        # the standard tile, 512 m at 2 m, quick look by IDW
        dict(name="tile_idw", kind="grid", survey="uniform", n=20_000, side_cm=51_200,
             cell_cm=200, nx=256, ny=256, method="idw", k=8, power=2.0, nbr=False),
        # the same tile by ordinary kriging with its variance
        dict(name="tile_krige", kind="grid", survey="uniform", n=20_000, side_cm=51_200,
             cell_cm=200, nx=256, ny=256, method="krige", k=16, model=0, nugget=0.25, sill=100.0,
             range=50.0),
        # the exponential model with a small nugget, an odd grid, a neighbourhood
        # that is no power of two, and the neighbour lists themselves
        dict(name="tile_odd_exp", kind="grid", survey="uniform", n=50_021, side_cm=66_430,
             cell_cm=130, nx=511, ny=333, method="krige", k=12, model=1, nugget=0.05, sill=80.0,
             range=40.0, nbr=True),
        # one survey line as it is logged: both grids from one call
        dict(name="line_both", kind="grid", survey="swath", lines=1, pings=3_001, cell_cm=50,
             nx=3_001, ny=692, method="both", k=32, k_idw=16, power=2.0, model=0, nugget=0.25,
             sill=100.0, range=50.0),
        # two lines, quick look by IDW over the whole box (a gap of coverage
        # between the lines)
        dict(name="swath_idw", kind="grid", survey="swath", lines=2, pings=4_000, cell_cm=50,
             nx=4_000, ny=1_692, method="idw", k=16, power=2.0, nbr=False),
        # the large survey: four 10 km lines, 0.5 m grid, IDW and kriging
        dict(name="swath_both", kind="grid", survey="swath", lines=4, pings=20_000, cell_cm=50,
             nx=20_000, ny=3_692, method="both", k=32, k_idw=16, power=2.0, model=0, nugget=0.25,
             sill=100.0, range=50.0),
        # the same end to end: soundings in pinned host memory, grids
        # delivered to pinned host memory
        dict(name="swath_host", kind="grid", survey="swath", lines=2, pings=4_001, cell_cm=50,
             nx=4_001, ny=1_692, method="host", k=32, k_idw=16, power=2.0, model=0, nugget=0.25,
             sill=100.0, range=50.0),
        # a planned batch of uneven tiles, IDW k = 16 and kriging k = 32 mixed
        dict(name="batch_mixed", kind="batch", tiles=96, mix=3, median_n=20_000),
        # a burst of uneven tiles through the serving queue, host to host
        dict(name="serve_burst", kind="serve", tiles=16, mix=5, median_n=20_000),
        # hole filling: the missing nodes of a gridded product, by both methods
        dict(name="holes_points", kind="points", nx=2_048, ny=2_048, cell_cm=200, frac=0.05,
             k=32, k_idw=16, power=2.0, model=0, nugget=0.25, sill=100.0, range=50.0),
        # row filling of a gridded product (rows halfway between its rows)
        dict(name="resample_rows", kind="resample", mode="rows", nx=8_192, ny=8_192, cell_cm=200,
             frac=0.05, method=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vgm(rng):
    if rng.random() < 0.7:
        return dict(model=0, nugget=round(rng.uniform(0.1, 1.0), 3), sill=round(rng.uniform(50.0, 150.0), 2),
                    range=round(rng.uniform(20.0, 120.0), 2))
    return dict(model=1, nugget=round(rng.uniform(0.05, 0.5), 3), sill=round(rng.uniform(50.0, 150.0), 2),
                range=round(rng.uniform(20.0, 80.0), 2))


def draw(rng):
    kind = rng.choice(["tile", "tile", "tile", "swath", "swath", "batch", "serve", "points", "resample"])
    if kind == "tile":
        n = _log(rng, 1_000, 400_000)
        cell = 2 * rng.randint(50, 200)
        nx, ny = _log(rng, 50, 1_100), _log(rng, 50, 1_100)
        c = dict(kind="grid", survey="uniform", n=n, side_cm=max(nx, ny) * cell, cell_cm=cell, nx=nx, ny=ny)
        method = rng.choice(["idw", "krige", "both"])
        if method == "idw":
            c.update(method="idw", k=rng.choice([8, 16, 16, 5, 32]),
                     power=rng.choice([2.0, 2.0, 2.0, 3.0, 1.5]), nbr=rng.random() < 0.2)
        elif method == "krige":
            c.update(method="krige", k=rng.choice([8, 16, 16, 32, 32, 12, 24]), nbr=rng.random() < 0.2, **_vgm(rng))
        else:
            c.update(method="both", k=32, k_idw=rng.choice([8, 16]), power=2.0, **_vgm(rng))
        return c
    if kind == "swath":
        lines, pings = rng.randint(1, 3), _log(rng, 500, 6_000)
        cell = rng.choice([50, 50, 100, 70])
        half = ALTITUDE_M * math.tan(math.radians(FAN_DEG))
        c = dict(kind="grid", survey="swath", lines=lines, pings=pings, cell_cm=cell,
                 nx=max(8, int(pings * PING_STEP_M * 100) // cell - rng.randint(0, 3)),
                 ny=int((2 * half + (lines - 1) * LINE_SPACING_M) * 100 / cell))
        method = rng.choice(["both", "both", "idw", "krige", "host"])
        c.update(method=method, k=16 if method == "idw" else rng.choice([32, 32, 32, 16]))
        if method != "krige":
            c.update(power=2.0)
        if method in ("both", "host"):
            c.update(k_idw=16)
        if method != "idw":
            c.update(**_vgm(rng))
        return c
    if kind == "batch":
        return dict(kind="batch", tiles=_log(rng, 8, 128), mix=rng.randint(10, 10_000),
                    median_n=_log(rng, 5_000, 40_000))
    if kind == "serve":
        return dict(kind="serve", tiles=_log(rng, 4, 24), mix=rng.randint(10, 10_000),
                    median_n=_log(rng, 5_000, 30_000))
    if kind == "points":
        return dict(kind="points", nx=_log(rng, 300, 3_000), ny=_log(rng, 300, 3_000),
                    cell_cm=2 * rng.randint(50, 150), frac=rng.choice([0.01, 0.05, 0.1]),
                    k=rng.choice([32, 32, 16]), k_idw=rng.choice([8, 16]), power=2.0, **_vgm(rng))
    return dict(kind="resample", mode=rng.choice(["rows", "grid", "points"]), nx=_log(rng, 500, 7_000),
                ny=_log(rng, 500, 7_000), cell_cm=2 * rng.randint(50, 150),
                frac=rng.choice([0.01, 0.05, 0.1]), method=rng.randint(0, 1))


# ------------------------------------------------------------------ inputs

def _gen(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    return g


def _rand(g, m, lo, hi):
    return torch.rand(m, generator=g, device=g.device, dtype=torch.float64) * (hi - lo) + lo


def _depth(g, x_m, y_m, noise_m=0.5):
    """Slope, twenty long-crested undulations of a few metres each, noise."""
    d = torch.full_like(x_m, 3500.0) + 0.01 * x_m
    wl, ang, ph, amp = (_rand(g, 20, *r).tolist()
                        for r in ((60.0, 500.0), (0.0, math.pi), (0.0, 6.2831853), (1.0, 6.0)))
    for w, a, p, s in zip(wl, ang, ph, amp):
        d += s * torch.sin(x_m * (math.cos(a) * 6.2831853 / w) + y_m * (math.sin(a) * 6.2831853 / w) + p)
    if noise_m > 0:
        d += noise_m * torch.randn(d.shape, generator=g, device=d.device, dtype=d.dtype)
    return d.float()


def _uniform(g, n, w_cm, h_cm):
    x = torch.randint(0, w_cm, (n,), generator=g, device="cuda", dtype=torch.int32)
    y = torch.randint(0, h_cm, (n,), generator=g, device="cuda", dtype=torch.int32)
    z = _depth(g, x.double() / 100, y.double() / 100)
    z[torch.rand(n, generator=g, device="cuda") < 0.002] = float("nan")
    return x, y, z


def _swath(g, lines, pings):
    theta = torch.linspace(-FAN_DEG, FAN_DEG, BEAMS, dtype=torch.float64, device="cuda") * (math.pi / 180)
    across = ALTITUDE_M * torch.tan(theta)
    half = float(across.max())
    px = torch.arange(pings, dtype=torch.float64, device="cuda") * PING_STEP_M
    xs, ys, zs = [], [], []
    sea = int(torch.randint(0, 1 << 30, (1,), generator=g, device="cuda"))
    for line in range(lines):
        x = px.repeat_interleave(BEAMS)
        y = (half + line * LINE_SPACING_M + across).repeat(pings)
        x = x + _rand(g, x.numel(), -1.0, 1.0)
        y = y + _rand(g, y.numel(), -1.0, 1.0)
        xc, yc = torch.floor(x * 100 + 0.5), torch.floor(y * 100 + 0.5)
        z = _depth(_gen(sea), xc / 100, yc / 100, 0.0)
        z += 0.5 * torch.randn(z.shape, generator=g, device="cuda")
        z[torch.rand(z.shape, generator=g, device="cuda") < 0.002] = float("nan")
        xs.append(xc.int())
        ys.append(yc.int())
        zs.append(z)
    return torch.cat(xs), torch.cat(ys), torch.cat(zs)


def _mix(case):
    """Tiles of uneven size: lognormal soundings, grid sides and cells of the
    survey mix, a fair coin between IDW k = 16 and kriging k = 32."""
    r = np.random.Generator(np.random.PCG64(case["mix"]))
    out = []
    for _ in range(case["tiles"]):
        n = int(np.clip(round(case["median_n"] * math.exp(r.standard_normal())), 1_000, 200_000))
        side, cell = int(r.choice(SIDES)), int(r.choice(CELLS_M)) * 100
        out.append(dict(n=n, side=side, cell=cell, method=int(r.integers(0, 2))))
    return out


def _variogram(case):
    return bg.variogram(case["model"], case["nugget"], case["sill"], case["range"])


def _product(case, seed):
    """A gridded depth product and the sorted indices of its missing nodes."""
    g = _gen(seed)
    nx, ny, cell = case["nx"], case["ny"], case["cell_cm"]
    x = torch.arange(nx, device="cuda", dtype=torch.float64).mul_(cell).add_(cell // 2) / 100
    y = torch.arange(ny, device="cuda", dtype=torch.float64).mul_(cell).add_(cell // 2) / 100
    z = _depth(g, x.repeat(ny), y.repeat_interleave(nx), 0.0)
    m = nx * ny
    gone = torch.zeros(m, dtype=torch.bool, device="cuda")
    gone[torch.randperm(m, generator=g, device="cuda")[:int(round(case["frac"] * m))]] = True
    return z, gone


def _node_xy(case, idx):
    cell = case["cell_cm"]
    return ((idx % case["nx"]) * cell + cell // 2).int(), ((idx // case["nx"]) * cell + cell // 2).int()


# ------------------------------------------------------------------- state

_CTX = []


def _ctx():
    if not _CTX:
        _CTX.append(bg.ctx_create(0))
    return _CTX[0]


class State:
    pass


def _soundings(case, seed):
    g = _gen(seed)
    if case["survey"] == "swath":
        return _swath(g, case["lines"], case["pings"])
    return _uniform(g, case["n"], case["nx"] * case["cell_cm"], case["ny"] * case["cell_cm"])


def _tiles(case, seed):
    out = []
    for i, t in enumerate(_mix(case)):
        span = t["side"] * t["cell"]
        out.append((t, _uniform(_gen(seed * 1_000_003 + i), t["n"], span, span)))
    return out


def prepare(case, seed):
    s = State()
    s.case, s.ctx = case, _ctx()
    dev = "cuda"
    kind = case["kind"]
    if kind == "grid":
        m = case["nx"] * case["ny"]
        s.xyz = _soundings(case, seed)
        if case["method"] == "host":
            s.xyz = tuple(t.cpu().pin_memory() for t in s.xyz)
            s.host = [torch.empty(m, pin_memory=True) for _ in range(3)]
        s.grid = bg.grid_create(s.ctx, 0, 0, case["cell_cm"], case["nx"], case["ny"])
        weakref.finalize(s, bg.grid_destroy, s.grid)
        s.out = {}
        if case["method"] in ("idw", "both", "host"):
            s.out["idw"] = torch.empty(m, device=dev)
        if case["method"] != "idw":
            s.out["depth"] = torch.empty(m, device=dev)
            s.out["var"] = torch.empty(m, device=dev)
            s.vgm = _variogram(case)
        if case.get("nbr"):
            s.out["nbr"] = torch.empty(m * case["k"], dtype=torch.int32, device=dev)
    elif kind == "batch":
        data = _tiles(case, seed)
        m = sum(t["side"] ** 2 for t, _ in data)
        mk = sum(t["side"] ** 2 for t, _ in data if t["method"] == 1)
        s.out = dict(depth=torch.empty(m, device=dev), var=torch.empty(mk, device=dev))
        tiles, at, atk = [], 0, 0
        for t, (x, y, z) in data:
            q = t["side"] ** 2
            d = dict(x_cm=x, y_cm=y, z_m=z, grid_spec=(0, 0, t["cell"], t["side"], t["side"]),
                     method=t["method"], k=32 if t["method"] else 16, depth_out=s.out["depth"][at:at + q])
            at += q
            if t["method"]:
                d["var_out"] = s.out["var"][atk:atk + q]
                atk += q
            tiles.append(d)
        s.batch = bg.batch_create(s.ctx, tiles)
        weakref.finalize(s, bg.batch_destroy, s.batch)
    elif kind == "serve":
        s.reqs = []
        for t, xyz in _tiles(case, seed):
            q = t["side"] ** 2
            s.reqs.append((t, [v.cpu().numpy() for v in xyz], np.empty(q, np.float32),
                           np.empty(q, np.float32) if t["method"] else None))
    elif kind == "points":
        z, gone = _product(case, seed)
        kept, holes = torch.nonzero(~gone).flatten(), torch.nonzero(gone).flatten()
        s.xyz = (*_node_xy(case, kept), z[kept])
        s.q = _node_xy(case, holes)
        m = holes.numel()
        s.out = dict(idw=torch.empty(m, device=dev), depth=torch.empty(m, device=dev),
                     var=torch.empty(m, device=dev))
        s.vgm = _variogram(case)
    else:
        z, gone = _product(case, seed)
        z[gone] = float("nan")
        s.src, cell, nx, ny = z, case["cell_cm"], case["nx"], case["ny"]
        s.spec = (0, 0, cell, nx, ny)
        if case["mode"] == "rows":      # halfway between the source's rows
            s.ospec = (0, cell // 2, cell, nx, ny - 1)
        elif case["mode"] == "grid":    # another origin and a finer cell
            oc = max(2, cell * 3 // 4 // 2 * 2)
            s.ospec = (cell // 3, cell // 5, oc, nx, ny)
        else:
            g = _gen(seed + 7)
            s.q = tuple(torch.randint(0, n * cell, (nx * ny,), generator=g, device=dev, dtype=torch.int32)
                        for n in (nx, ny))
        m = nx * ny if case["mode"] == "points" else s.ospec[3] * s.ospec[4]
        s.out = dict(depth=torch.empty(m, device=dev), how=torch.empty(m, dtype=torch.int8, device=dev))
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "grid":
        h = bg.soundings_upload(s.ctx, *s.xyz)
        o, k, method = s.out, case["k"], case["method"]
        if method == "idw":
            bg.interp_idw(h, s.grid, k, case["power"], o["idw"], o.get("nbr"))
        elif method == "krige":
            bg.interp_okrige(h, s.grid, k, s.vgm, o["depth"], o["var"], o.get("nbr"))
        elif method == "both":
            bg.interp_idw_okrige(h, s.grid, case["k_idw"], case["power"], k, s.vgm, o["idw"],
                                 o["depth"], o["var"])
        else:
            bg.interp_idw_okrige_host(h, s.grid, case["k_idw"], case["power"], k, s.vgm, o["idw"],
                                      o["depth"], o["var"], *s.host)
        bg.soundings_destroy(h)
        return dict(zip(("idw", "depth", "var"), s.host)) if method == "host" else o
    if kind == "batch":
        bg.batch_run(s.batch)
        return s.out
    if kind == "serve":
        tickets = [bg.submit(s.ctx, *xyz, (0, 0, t["cell"], t["side"], t["side"]), t["method"],
                             32 if t["method"] else 16, depth, var)
                   for t, xyz, depth, var in s.reqs]
        for t in tickets:
            bg.wait(s.ctx, t)
        return [[depth] if var is None else [depth, var] for _, _, depth, var in s.reqs]
    if kind == "points":
        h = bg.soundings_upload(s.ctx, *s.xyz)
        bg.interp_idw_points(h, *s.q, case["k_idw"], case["power"], s.out["idw"])
        bg.interp_okrige_points(h, *s.q, case["k"], s.vgm, s.out["depth"], s.out["var"])
        bg.soundings_destroy(h)
        return s.out
    if case["mode"] == "points":
        bg.resample_points(s.src, s.spec, case["method"], *s.q, s.out["depth"], s.out["how"])
    else:
        bg.resample_grid(s.src, s.spec, case["method"], s.ospec, s.out["depth"], s.out["how"])
    return s.out


# -------------------------------------------------------------------- work

def _node_flops(method, k):
    """Per node: weights and sums of IDW; the variogram matrix, one symmetric
    factorization, two solves and a residual of the kriging system."""
    if method == 0:
        return 8.0 * k
    n = k - 1
    return n ** 3 / 3.0 + 2 * (2.0 * n * n) + 2.0 * n * n + 12.0 * (n * (n + 1) / 2 + n)


def work(case):
    kind = case["kind"]
    if kind == "grid":
        m = case["nx"] * case["ny"]
        n = case["lines"] * case["pings"] * BEAMS if case["survey"] == "swath" else case["n"]
        outs = {"idw": 1, "krige": 2}.get(case["method"], 3)
        fl = 0.0
        if case["method"] != "krige":
            fl += _node_flops(0, case.get("k_idw", case["k"])) * m
        if case["method"] != "idw":
            fl += _node_flops(1, case["k"]) * m
        return dict(bytes=12.0 * n + 4.0 * m * (outs + (case["k"] if case.get("nbr") else 0)), flops=fl)
    if kind in ("batch", "serve"):
        b = f = 0.0
        for t in _mix(case):
            m = t["side"] ** 2
            b += 12.0 * t["n"] + 4.0 * m * (1 + t["method"])
            f += m * _node_flops(t["method"], 32 if t["method"] else 16)
        return dict(bytes=b, flops=f)
    m = case["nx"] * case["ny"]
    if kind == "points":
        q = m * case["frac"]
        return dict(bytes=12.0 * (m - q) + 2 * 8.0 * q + 12.0 * q,
                    flops=q * (_node_flops(0, case["k_idw"]) + _node_flops(1, case["k"])))
    per = 9.0 + (8.0 if case["mode"] == "points" else 0.0)
    return dict(bytes=per * m, flops=m * (10.0 if case["method"] == 0 else 40.0))


# ------------------------------------------------------------------- exact

def _neighbours(x, y, valid, qx, qy, k):
    """The k nearest valid soundings of each query: (d2, index) ascending, by
    brute force over blocks of queries, against the soundings of a window
    around each block that is widened until it must hold them all."""
    idx = torch.nonzero(valid).flatten()
    sx, sy = x[idx].long(), y[idx].long()
    order = torch.argsort(sx)
    idx, sx, sy = idx[order], sx[order], sy[order]
    bits = max(1, int(x.numel() - 1).bit_length())
    m = qx.numel()
    out_d = torch.empty(m, k, dtype=torch.int64, device=qx.device)
    out_i = torch.empty(m, k, dtype=torch.int64, device=qx.device)
    qx, qy = qx.long(), qy.long()
    side = 3_200
    block = (qy.div(side, rounding_mode="floor") * (1 << 24)) + qx.div(side, rounding_mode="floor")
    perm = torch.argsort(block)
    counts = torch.unique_consecutive(block[perm], return_counts=True)[1].tolist()
    at = 0
    step = 1 << 12
    for c in counts:
        for lo in range(at, at + c, step):
            p = perm[lo:min(lo + step, at + c)]
            bx, by = qx[p], qy[p]
            x0, x1, y0, y1 = (int(v) for v in (bx.min(), bx.max(), by.min(), by.max()))
            margin = 800
            while True:
                a = int(torch.searchsorted(sx, x0 - margin))
                b = int(torch.searchsorted(sx, x1 + margin, right=True))
                sel = torch.nonzero((sy[a:b] >= y0 - margin) & (sy[a:b] <= y1 + margin)).flatten() + a
                whole = sel.numel() == sx.numel()
                if sel.numel() >= k or whole:
                    cx, cy, ci = sx[sel], sy[sel], idx[sel]
                    rows = max(1, min(p.numel(), (1 << 26) // max(1, sel.numel())))
                    keys = torch.cat([torch.topk(
                        (((bx[r:r + rows, None] - cx) ** 2 + (by[r:r + rows, None] - cy) ** 2) << bits) + ci,
                        k, dim=1, largest=False, sorted=True)[0] for r in range(0, p.numel(), rows)])
                    if whole or int(keys[:, -1].max() >> bits) <= margin * margin:
                        break
                margin *= 2
            out_d[p], out_i[p] = keys >> bits, keys & ((1 << bits) - 1)
        at += c
    return out_d, out_i


def _exact_idw(d2, zi, power):
    z = zi.double()
    d = d2.double()
    w = (d[:, :1] / d) ** (0.5 * power)
    v = (w * z).sum(1) / w.sum(1)
    return torch.where(d2[:, 0] == 0, z[:, 0], v)


def _gamma(case, h):
    c0, c = case["nugget"], case["sill"] - case["nugget"]
    t = h / case["range"]
    if case["model"] == 0:
        return torch.where(t < 1, c0 + c * (1.5 * t - 0.5 * t ** 3), torch.full_like(t, case["sill"]))
    return c0 - c * torch.expm1(-t)


def _exact_krige(case, x, y, d2, ii, zi):
    m, k = ii.shape
    depth = torch.empty(m, dtype=torch.float64, device=ii.device)
    var = torch.empty_like(depth)
    eye = torch.eye(k, dtype=torch.bool, device=ii.device)
    f32 = {q: float(np.float32(case[q])) for q in ("nugget", "sill", "range")} | {"model": case["model"]}
    for lo in range(0, m, 1 << 16):
        s = slice(lo, min(lo + (1 << 16), m))
        px, py = x[ii[s]].double() / 100, y[ii[s]].double() / 100
        h = torch.hypot(px[:, :, None] - px[:, None, :], py[:, :, None] - py[:, None, :])
        A = torch.ones(h.shape[0], k + 1, k + 1, dtype=torch.float64, device=ii.device)
        A[:, :k, :k] = _gamma(f32, h).masked_fill(eye, 0.0)
        A[:, k, k] = 0.0
        g0 = _gamma(f32, d2[s].double().sqrt() / 100)
        g0 = torch.where(d2[s] == 0, torch.zeros_like(g0), g0)
        b = torch.cat([g0, torch.ones_like(g0[:, :1])], 1)
        lam = torch.linalg.solve(A, b)
        depth[s] = (lam[:, :k] * zi[s].double()).sum(1)
        var[s] = (lam * b).sum(1)
    return depth, var


def _exact_grid(case, x, y, z, qx, qy, want):
    valid = ~torch.isnan(z)
    d2, ii = _neighbours(x, y, valid, qx, qy, case["k"])
    zi = z[ii]
    out = {}
    if "idw" in want:
        k = case.get("k_idw", case["k"])
        out["idw"] = _exact_idw(d2[:, :k], zi[:, :k], case["power"])
    if "depth" in want:
        out["depth"], out["var"] = _exact_krige(case, x, y, d2, ii, zi)
    if "nbr" in want:
        out["nbr"] = ii.int().flatten()
    return out


def _exact_resample(case, seed):
    s = prepare(case, seed)
    nx, ny, cell = case["nx"], case["ny"], case["cell_cm"]
    src = s.src.double().view(ny, nx)
    if case["mode"] == "points":
        u, v = (q.double() - cell // 2 for q in s.q)
    else:
        ox, oy, oc, onx, ony = s.ospec
        u = (torch.arange(onx, device="cuda", dtype=torch.float64) * oc + ox + oc // 2 - cell // 2).repeat(ony)
        v = (torch.arange(ony, device="cuda", dtype=torch.float64) * oc + oy + oc // 2 - cell // 2
             ).repeat_interleave(onx)
    out = torch.empty_like(u)
    for lo in range(0, u.numel(), 1 << 22):
        q = slice(lo, min(lo + (1 << 22), u.numel()))
        a, b = u[q], v[q]
        inside = (a >= 0) & (a <= (nx - 1) * cell) & (b >= 0) & (b <= (ny - 1) * cell)
        i = torch.floor(a / cell).clamp(0, nx - 2).long()
        j = torch.floor(b / cell).clamp(0, ny - 2).long()
        t, r = a / cell - i, b / cell - j

        def corner(wx, wy, di, dj):
            w = wx * wy
            p = src[(j + dj).clamp(0, ny - 1), (i + di).clamp(0, nx - 1)]
            return torch.where(w != 0, w * p, torch.zeros_like(p))

        f = sum(corner(wx, wy, di, dj) for di, wx in ((0, 1 - t), (1, t)) for dj, wy in ((0, 1 - r), (1, r)))
        if case["method"] == 1:
            def cr(e):
                return (0.5 * (-e + 2 * e ** 2 - e ** 3), 0.5 * (2 - 5 * e ** 2 + 3 * e ** 3),
                        0.5 * (e + 4 * e ** 2 - 3 * e ** 3), 0.5 * (e ** 3 - e ** 2))
            c = sum(corner(wx, wy, di - 1, dj - 1) for di, wx in enumerate(cr(t)) for dj, wy in enumerate(cr(r)))
            f = torch.where(torch.isnan(c), f, c)
        out[q] = torch.where(inside, f, torch.full_like(f, float("nan")))
    return dict(depth=out, how=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "grid":
        m = case["nx"] * case["ny"]
        if m * (0.1 if case["method"] == "idw" else (case["k"] / 32) ** 2) > 2.5e6:
            return None  # over about 20 seconds
        x, y, z = _soundings(case, seed)
        cell = case["cell_cm"]
        want = {"idw": ["idw"], "krige": ["depth"], "both": ["idw", "depth"], "host": ["idw", "depth"]}[case["method"]]
        if case.get("nbr"):
            want = want + ["nbr"]
        qx, qy = _node_xy(case, torch.arange(m, device="cuda"))
        return _exact_grid(case, x, y, z, qx, qy, want)
    if kind == "points":
        z, gone = _product(case, seed)
        if case["nx"] * case["ny"] * case["frac"] > 1e6:
            return None
        kept, holes = torch.nonzero(~gone).flatten(), torch.nonzero(gone).flatten()
        return _exact_grid(case, *_node_xy(case, kept), z[kept], *_node_xy(case, holes), ["idw", "depth"])
    if kind == "resample":
        return _exact_resample(case, seed)
    if kind == "serve":
        out, left = [], 1_000_000  # nodes by kriging that fit the time
        for t, (x, y, z) in _tiles(case, seed):
            m = t["side"] ** 2
            cost = m if t["method"] else m // 10
            if cost > left:
                out.append([None, None] if t["method"] else [None])
                continue
            left -= cost
            c = dict(nx=t["side"], ny=t["side"], cell_cm=t["cell"], k=32 if t["method"] else 16, power=2.0,
                     model=0, nugget=0.25, sill=100.0, range=50.0)
            qx, qy = _node_xy(c, torch.arange(m, device="cuda"))
            r = _exact_grid(c, x, y, z, qx, qy, ["depth"] if t["method"] else ["idw"])
            out.append([r["depth"], r["var"]] if t["method"] else [r["idw"]])
        return out
    return None  # a batch's grids come whole, and all of them take over 20 seconds
