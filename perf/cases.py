"""The work that a program has this library do, through its public entry points, with sizes, options and inputs.

listed() names the cases and says what each stands for; draw() gives more of the same ranges.  Maps are 0.05 m occupancy
grids (a walled room, an office of rooms and corridors, a warehouse of identical shelves), hypotheses are free cells with
0.2 m of clearance, and a scan is marched from a pose near one hypothesis, with range noise, short returns and dropouts.

Kinds of work:
  locate    one relocalization (hypotheses, scan -> pose and scores), blocking from host arrays ("host") or from a scan
            already on the GPU ("device"); with "update" the map's tables are rebuilt from a new grid first
  batch     several requests in one call; with "resident" the context keeps the synthesized scans of its maps
  update    a new grid for a loaded map: exact distance transform, likelihood field, occupancy
  edt       the distance transform into the caller's memory, without a context or an allocation
  synth     synthesized scans with hit cells of given cells
  sample    positional hypotheses from the occupancy grid (the traversability-constrained RRT)
"""
import math

import numpy as np
import torch

import paper_2511_01219_gb300 as relo

RES = 0.05
FREE, OCC, UNKNOWN = 0, 100, -1
BATCH, LOCAL, TAU = 200, 20, 0.95   # the library's defaults: survivors per batch, local top-k, early-termination score
D_MAX = 2.0
MAX_BEAMS, MAX_NS = 2048, 8192


# ---- cases -------------------------------------------------------------------------------------------------------------

def locate(name, side, plan, beams, ns, orient, hyps, topk, max_range, how="host", update=False, early=False, icp=0,
           coarse="smad"):
    c = {"kind": "locate", "w": side[0], "h": side[1], "plan": plan, "beams": beams, "ns": ns, "orient": orient,
         "hyps": hyps, "topk": topk, "max_range": max_range, "how": how, "update": update, "early": early, "icp": icp,
         "coarse": coarse}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a small robot in one room: the smallest call, a few launches and their latency (64^2, 200 hypotheses)
        locate("room call", (64, 64), "room", 360, 504, 72, 200, 16, 10.0),
        # one floor of an office, the ordinary call: 270 degree scan, every survivor scored
        locate("office call", (1024, 1024), "office", 1081, 1440, 360, 5000, 256, 25.0),
        # the same floor as a robot's loop runs it: early termination, and the best poses refined by ICP and scored again
        locate("office loop with refinement", (1024, 1024), "office", 1081, 1440, 360, 5000, 256, 25.0, early=True, icp=10),
        # an odd-sized map and a coarse scanner, ranked beam by beam (CAER), scan on the GPU
        locate("beam-wise ranking", (777, 603), "office", 541, 1080, 360, 2500, 256, 25.0, how="device", coarse="caer"),
        # a warehouse whose map has changed: tables rebuilt, then a full-circle scan against 20000 hypotheses
        locate("warehouse step", (4096, 4096), "warehouse", 1440, 1440, 720, 20000, 1024, 25.0, how="device", update=True),
        # a fleet's requests in one call: maps, scanners and fields of view differ
        {"name": "mixed batch", "kind": "batch", "maps": 4, "requests": 16, "lo": 512, "hi": 2048, "orient": 360,
         "hyps": 8000, "topk": 512, "resident": False},
        # a server's requests against maps whose synthesized scans it keeps
        {"name": "resident batch", "kind": "batch", "maps": 4, "requests": 16, "lo": 512, "hi": 2048, "orient": 360,
         "hyps": 8000, "topk": 256, "resident": True},
        # a door has opened on an office floor; a large warehouse is loaded again
        {"name": "office map update", "kind": "update", "w": 1024, "h": 1024, "plan": "office"},
        {"name": "large map update", "kind": "update", "w": 4001, "h": 3500, "plan": "office"},
        # the distance transform in a control loop that may not allocate
        {"name": "distance transform", "kind": "edt", "w": 1000, "h": 777, "plan": "office"},
        # synthesized scans of many cells, for a user's own matching
        {"name": "synthesized scans", "kind": "synth", "w": 2048, "h": 2048, "plan": "office", "beams": 1081, "ns": 1440,
         "cells": 6000, "max_range": 25.0},
        # hypotheses of a floor, before its first relocalization
        {"name": "hypothesis sampling", "kind": "sample", "w": 1024, "h": 1024, "plan": "office", "rho": 0.6},
    ]


def log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def sensor(rng, orient):
    """(beams, N_s): N_s a multiple of the orientation count with beams <= N_s <= 2 beams."""
    while True:
        beams = rng.choice((361, 541, 720, 1081, 1440, log_int(rng, 200, 2000)))
        lo, hi = -(-beams // orient), min(2 * beams, MAX_NS) // orient
        if hi >= lo:
            return beams, orient * rng.randint(lo, hi)


def draw(rng):
    kind = rng.choice(("locate",) * 5 + ("batch", "batch", "update", "edt", "synth", "sample"))
    plan = rng.choice(("office", "warehouse"))
    if kind == "locate":
        orient = rng.choice((72, 120, 180, 360, 360))
        beams, ns = sensor(rng, orient)
        room = rng.random() < 0.2
        w, h = (rng.randint(64, 160),) * 2 if room else (log_int(rng, 256, 3000), log_int(rng, 256, 3000))
        coarse = "caer" if rng.random() < 0.15 else "smad"
        hyps = log_int(rng, 100, 600 if room else 3000 if coarse == "caer" else 16000)
        early = rng.random() < 0.4
        return locate(None, (w, h), "room" if room else plan, beams, ns, orient, hyps, log_int(rng, 16, 900),
                      rng.choice((8.0, 12.5, 25.0)), how=rng.choice(("host", "device")), update=rng.random() < 0.3,
                      early=early, icp=rng.choice((0, 5, 10)) if early else 0, coarse=coarse)
    if kind == "batch":
        lo = log_int(rng, 300, 900)
        return {"kind": "batch", "maps": rng.randint(1, 4), "requests": rng.randint(2, 14), "lo": lo,
                "hi": lo + rng.randint(0, 900), "orient": rng.choice((180, 360)), "hyps": log_int(rng, 500, 8000),
                "topk": log_int(rng, 50, 512), "resident": rng.random() < 0.5}
    if kind == "update":
        return {"kind": "update", "w": log_int(rng, 100, 3700), "h": log_int(rng, 100, 3700), "plan": plan}
    if kind == "edt":
        return {"kind": "edt", "w": log_int(rng, 60, 1024), "h": log_int(rng, 60, 1024), "plan": plan}
    if kind == "synth":
        beams, ns = sensor(rng, 90)
        return {"kind": "synth", "w": log_int(rng, 200, 2048), "h": log_int(rng, 200, 2048), "plan": plan, "beams": beams,
                "ns": ns, "cells": log_int(rng, 10, 6000), "max_range": rng.choice((8.0, 12.5, 25.0))}
    return {"kind": "sample", "w": log_int(rng, 150, 1000), "h": log_int(rng, 150, 1000), "plan": plan,
            "rho": rng.choice((0.6, 0.8, 1.0))}


# ---- maps, scans and hypotheses ----------------------------------------------------------------------------------------

def grid_of(plan, w, h, rng):
    """int8 [h, w]: 0 free, 100 occupied, -1 unknown."""
    g = np.zeros((h, w), np.int8)
    if plan == "room":
        g[[0, -1], :] = OCC
        g[:, [0, -1]] = OCC
        for _ in range(6):
            bw, bh = (int(v) for v in rng.integers(2, 9, 2))
            x, y = int(rng.integers(2, w - 2 - bw)), int(rng.integers(2, h - 2 - bh))
            g[y:y + bh, x:x + bw] = OCC
        return g
    if plan == "warehouse":   # 1 m shelves, 3 m aisles, a cross aisle every 20 m at most, perimeter walls, a few pillars
        g[[0, -1], :] = OCC
        g[:, [0, -1]] = OCC
        edge = max(8, min(80, w // 8, h // 8))
        run = max(10, min(400, (w - 2 * edge - 50) // 2))
        for y in range(edge, h - edge - 20, 80):
            for x in range(edge, w - edge - run + 1, run + 50):
                g[y:y + 20, x:x + run] = OCC
        for _ in range(8):
            x, y = int(rng.integers(2, w - 8)), int(rng.integers(2, edge - 5))
            g[y:y + 6, x:x + 6] = OCC
        return g
    # office: an unknown band outside, rooms of 4 to 9 m split off by 1.5 m corridors, 0.9 m doors, furniture
    band = max(1, round(0.0075 * min(w, h)))
    g[:] = UNKNOWN
    g[band:h - band, band:w - band] = FREE
    g[[band, h - band - 1], band:w - band] = OCC
    g[band:h - band, [band, w - band - 1]] = OCC
    rooms, todo = [], [(band + 1, band + 1, w - band - 1, h - band - 1)]

    def wall(a, lo, hi, upright):
        line = g[lo:hi, a] if upright else g[a, lo:hi]
        line[:] = OCC
        if hi - lo > 22:
            d = int(rng.integers(2, hi - lo - 20))
            line[d:d + 18] = FREE

    while todo:
        x0, y0, x1, y1 = todo.pop()
        bw, bh = x1 - x0, y1 - y0
        if max(bw, bh) <= 180 or max(bw, bh) < 190:
            rooms.append((x0, y0, x1, y1))
        elif bw >= bh:
            s = int(rng.integers(x0 + 80, x1 - 80 - 30 + 1))
            wall(s, y0, y1, True)
            wall(s + 29, y0, y1, True)
            todo += [(x0, y0, s, y1), (s + 30, y0, x1, y1)]
        else:
            s = int(rng.integers(y0 + 80, y1 - 80 - 30 + 1))
            wall(s, x0, x1, False)
            wall(s + 29, x0, x1, False)
            todo += [(x0, y0, x1, s), (x0, s + 30, x1, y1)]
    for x0, y0, x1, y1 in rooms:
        for _ in range(int(rng.integers(0, 4))):
            bw, bh = (int(v) for v in rng.integers(8, 30, 2))
            if x1 - x0 - bw > 12 and y1 - y0 - bh > 12:
                x, y = int(rng.integers(x0 + 4, x1 - bw - 4)), int(rng.integers(y0 + 4, y1 - bh - 4))
                g[y:y + bh, x:x + bw] = OCC
    return g


def free_cells(grid_t, n, rng):
    """n distinct cells (cx, cy) with 0.2 m of clearance (free space if there are too few), in row order, int32 numpy."""
    blocked = (grid_t != FREE).to(torch.float16)[None, None]
    near = torch.nn.functional.max_pool2d(blocked, 9, 1, 4)[0, 0]
    cells = torch.nonzero(near == 0)
    if len(cells) < n:
        cells = torch.nonzero(grid_t == FREE)
    pick = np.sort(rng.choice(len(cells), min(n, len(cells)), replace=False))
    return np.ascontiguousarray(cells[torch.from_numpy(pick).to(cells.device)].flip(1).cpu().numpy().astype(np.int32))


def angles_of(beams, ns):
    j = np.arange(beams, dtype=np.float64) - beams // 2
    a = j * (2.0 * math.pi / ns)
    return ((a + math.pi) % (2.0 * math.pi) - math.pi).astype(np.float32)


def scan_of(grid_t, cells, beams, ns, orient, max_range, rng):
    """float32 ranges of a scan from a pose within 0.25 m of a hypothesis: 10 % short returns, 2 cm noise, 5 % dropouts."""
    h, w = grid_t.shape
    c = cells[int(rng.integers(len(cells)))]
    off = rng.uniform(-0.25, 0.25, 2) / RES
    x, y = c[0] + 0.5 + off[0], c[1] + 0.5 + off[1]
    if not (0 <= x < w and 0 <= y < h) or int(grid_t[int(y), int(x)]) != FREE:
        x, y = c[0] + 0.5, c[1] + 0.5
    th = int(rng.integers(orient)) * 2.0 * math.pi / orient
    a = torch.from_numpy(angles_of(beams, ns).astype(np.float64) + th).cuda()
    t = torch.arange(1, int(max_range / RES * 4) + 1, device="cuda", dtype=torch.float64) * 0.25
    px = torch.floor(x + torch.cos(a)[:, None] * t).to(torch.int64)
    py = torch.floor(y + torch.sin(a)[:, None] * t).to(torch.int64)
    inside = (px >= 0) & (py >= 0) & (px < w) & (py < h)
    occ = inside & (grid_t[py.clamp(0, h - 1), px.clamp(0, w - 1)] >= 65)
    first = torch.where(occ, t, torch.full_like(t, math.inf)).amin(1)
    z = np.minimum(first.cpu().numpy() * RES, max_range)
    ret = z < max_range
    short = ret & (rng.random(beams) < 0.10) & (z > 0.1)
    z = np.where(short, rng.uniform(0.1, np.maximum(z, 0.11)), z) + np.where(ret, rng.normal(0.0, 0.02, beams), 0.0)
    z = np.clip(z, 1e-3, max_range)
    z[rng.random(beams) < 0.05] = max_range
    return z.astype(np.float32)


def rng_of(seed):
    return np.random.default_rng([2511, int(seed)])


def to_gpu(a):
    return torch.from_numpy(a).cuda()


def inputs(case, seed):
    """grid (numpy and on the GPU), hypothesis cells, angles, ranges."""
    rng = rng_of(seed)
    g = grid_of(case["plan"], case["w"], case["h"], rng)
    gt = to_gpu(g)
    cells = free_cells(gt, case["hyps"], rng)
    z = scan_of(gt, cells, case["beams"], case["ns"], case["orient"], case["max_range"], rng)
    return g, gt, cells, angles_of(case["beams"], case["ns"]), z


def batch_inputs(case, seed):
    """maps [(grid, cells)] and requests [(map, ranges, angles, max_range, topk)]; sizes and scanners by the seed."""
    rng = rng_of(seed)
    shape = rng_of(4242)   # the fleet's sizes and scanners are the case's, not the seed's
    maps, reqs = [], []
    for i in range(case["maps"]):
        w, h = (int(v) for v in shape.integers(case["lo"], case["hi"] + 1, 2))
        g = grid_of(("office", "warehouse")[i % 2], w, h, rng)
        gt = to_gpu(g)
        maps.append((g, gt, free_cells(gt, case["hyps"] * (1 + 2 * i) // 8 + 1, rng)))
    for r in range(case["requests"]):
        g, gt, cells = maps[r % case["maps"]]
        beams = int(shape.choice((541, 720, 1081, 1440)))
        o = case["orient"]
        ns = o * int(shape.integers(-(-beams // o), 2 * beams // o + 1))
        z = scan_of(gt, cells, beams, ns, o, 25.0, rng)
        reqs.append((r % case["maps"], z, angles_of(beams, ns), 25.0, max(1, case["topk"] // (1 + r % 2))))
    return maps, reqs


# ---- the calls ---------------------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "locate":
        g, gt, cells, angles, z = inputs(case, seed)
        ctx = relo.Relo(n_orient=case["orient"], topk=case["topk"], early_stop=int(case["early"]), icp_iters=case["icp"],
                        coarse_metric=relo.COARSE_CAER if case["coarse"] == "caer" else relo.COARSE_SMAD)
        mid = ctx.load_map_dev(gt, RES)
        ctx.set_hypotheses_cells_dev(mid, to_gpu(cells))
        k = min(case["topk"], len(cells))
        return {"case": case, "ctx": ctx, "map": mid, "grid": gt, "angles": angles, "ranges": z, "ranges_t": to_gpu(z),
                "result_t": torch.zeros(relo.RESULT_BYTES, dtype=torch.uint8, device="cuda"),
                "scores": torch.empty((k, case["orient"]), dtype=torch.float32, device="cuda"),
                "numerators": torch.empty(len(cells), dtype=torch.int64, device="cuda")}
    if kind == "batch":
        maps, reqs = batch_inputs(case, seed)
        ctx = relo.Relo(n_orient=case["orient"], early_stop=0, scan_cache_bytes=(8 << 30) if case["resident"] else 0)
        ids = []
        for g, gt, cells in maps:
            ids.append(ctx.load_map_dev(gt, RES))
            ctx.set_hypotheses_cells_dev(ids[-1], to_gpu(cells))
        items = [(ids[m], z, a, r, min(k, len(maps[m][2]))) for m, z, a, r, k in reqs]
        if case["resident"]:
            ctx.relocalize_batch(items)   # a server has seen its sensors before
        return {"case": case, "ctx": ctx, "items": items,
                "scores": torch.empty((items[0][4], case["orient"]), dtype=torch.float32, device="cuda")}
    if kind == "update":
        g = to_gpu(grid_of(case["plan"], case["w"], case["h"], rng_of(seed)))
        ctx = relo.Relo()
        return {"case": case, "ctx": ctx, "map": ctx.load_map_dev(torch.zeros_like(g), RES), "grid": g}
    if kind == "edt":
        g = to_gpu(grid_of(case["plan"], case["w"], case["h"], rng_of(seed)))
        return {"case": case, "lib": relo.lib(), "grid": g, "d2": torch.empty(g.shape, dtype=torch.int32, device="cuda")}
    if kind == "synth":
        rng = rng_of(seed)
        g = to_gpu(grid_of(case["plan"], case["w"], case["h"], rng))
        ctx = relo.Relo(n_orient=0)   # every direction of the beam grid
        cells = to_gpu(free_cells(g, case["cells"], rng))
        return {"case": case, "ctx": ctx, "map": ctx.load_map_dev(g, RES), "cells": cells,
                "angles": angles_of(case["beams"], case["ns"])}
    rng = rng_of(seed)
    g = grid_of(case["plan"], case["w"], case["h"], rng)
    start = free_cells(to_gpu(g), 1, rng)[0]
    return {"case": case, "ctx": relo.Relo(), "grid": g, "p0": ((start[0] + 0.5) * RES, (start[1] + 0.5) * RES),
            "seed": int(rng.integers(1 << 30))}


WHOLE = ("hyp", "m", "n_batches", "status", "smad_num", "n_smad_evals", "n_tam_evals")


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "locate":
        ctx = s["ctx"]
        if case["update"]:
            ctx.update_map_dev(s["map"], s["grid"])
        if case["how"] == "host":
            r = ctx.relocalize(s["map"], s["ranges"], s["angles"], case["max_range"])
        else:
            ctx.relocalize_dev(s["map"], s["ranges_t"], s["angles"], case["max_range"], s["result_t"])
            r = relo.result_from_bytes(bytes(s["result_t"].cpu().numpy()))
        out = {k: int(getattr(r, k)) for k in WHOLE}
        out.update(x=r.x, y=r.y, theta=r.theta, smad=r.smad, tam=r.tam)
        out["scores"] = ctx.stage(relo.STAGE_TAM, s["scores"])
        out["numerators"] = ctx.stage(relo.STAGE_SMAD_NUM, s["numerators"])
        return out
    if kind == "batch":
        got = s["ctx"].relocalize_batch(s["items"])
        return {"whole": np.array([[getattr(r, k) for k in WHOLE] for r in got], np.int64),
                "pose": np.array([[r.x, r.y, r.theta, r.smad] for r in got]),
                "tam": np.array([r.tam for r in got], np.float32),
                "scores": s["ctx"].stage(relo.STAGE_TAM, s["scores"])}
    if kind == "update":
        s["ctx"].update_map_dev(s["map"], s["grid"])
        d2, field, occ = s["ctx"].map_tables(s["map"], s["grid"].shape)
        return {"d2": d2, "field": field, "occupied": occ}
    if kind == "edt":
        h, w = s["grid"].shape
        rc = s["lib"].relo_edt_noalloc(s["grid"].data_ptr(), w, h, s["d2"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if rc != relo.OK:
            raise relo.ReloError(rc, "relo_edt_noalloc")
        return s["d2"]
    if kind == "synth":
        ranges, hits = s["ctx"].synth_scans(s["map"], s["cells"], s["angles"], case["max_range"], case["ns"])
        return {"ranges": ranges, "hits": hits}
    xy, rounds, nodes = s["ctx"].rrt_sample(s["grid"], RES, s["p0"], case["rho"], seed=s["seed"])
    out = np.zeros((int(case["w"] * case["h"] * RES * RES / case["rho"] ** 2) + case["w"] + case["h"] + 16, 2))
    out[:len(xy)] = xy   # at most one representative per voxel; rows of zeros follow the last
    return {"xy": out, "count": len(xy), "rounds": rounds, "nodes": nodes}


def work(case):
    """Bytes: the grid, or the tables that a call reads, and what it returns, once each.  Operations: per beam of a scored pose
    an add, a compare and two sums; per ray of the ranking a sum; per cell of a distance transform a few."""
    kind = case["kind"]
    if kind == "locate":
        cells, k = case["w"] * case["h"], min(case["topk"], case["hyps"])
        poses, rays = k * case["orient"], case["hyps"] * case["ns"]
        per = 3 * case["beams"] if case["coarse"] == "caer" else 4
        b = cells * (7 if case["update"] else 2) + 24 * case["hyps"] + 4 * poses
        return {"bytes": b, "flops": 4 * poses * case["beams"] + rays + case["hyps"] * case["orient"] * per}
    if kind == "batch":
        r, side = case["requests"], (case["lo"] + case["hi"]) / 2
        poses = r * case["topk"] * 3 // 4 * case["orient"]
        return {"bytes": case["maps"] * side * side * 2 + 24 * case["hyps"] * r // 2 + 4 * poses,
                "flops": 4 * poses * 945 + r * case["hyps"] // 2 * (1400 + 4 * case["orient"])}
    cells = case["w"] * case["h"]
    if kind == "update":
        return {"bytes": cells * (1 + 4 + 4 + 1), "flops": 8 * cells}
    if kind == "edt":
        return {"bytes": cells * 5, "flops": 8 * cells}
    if kind == "synth":
        n = case["cells"] * case["ns"]
        return {"bytes": cells / 8 + 8 * case["cells"] + 8 * n, "flops": 40 * n}
    points = cells * RES * RES / case["rho"] ** 2 * 60   # about 60 rounds of one point per voxel
    return {"bytes": cells * 5 + 8 * points, "flops": points * 200}


# ---- the same in 64 bits -----------------------------------------------------------------------------------------------

def directions(ns):
    a = 2.0 * math.pi * np.arange(ns, dtype=np.float64) / ns
    return to_gpu(np.rint(np.stack([np.cos(a), np.sin(a)], 1) * 2.0 ** 30).astype(np.int64))


def cast_sums(gt, cells, ns, max_range):
    """int64 [n, ns] synthesized Q16 ranges: cell by cell from each cell centre, in the order of the grid-line crossings."""
    h, w = gt.shape
    occ = (gt >= 65).reshape(-1)
    lim = (round(max_range * 65536.0 / RES) ** 2) >> 32
    D = directions(ns)
    out = torch.zeros((len(cells), ns), dtype=torch.int64, device="cuda")
    for lo in range(0, len(cells), 4000):
        c = to_gpu(cells[lo:lo + 4000]).to(torch.int32)
        n = len(c)
        idx = torch.arange(n * ns, device="cuda")
        hx, hy = c[:, 0].repeat_interleave(ns), c[:, 1].repeat_interleave(ns)
        dx, dy = D[:, 0].repeat(n), D[:, 1].repeat(n)
        ax, ay = dx.abs(), dy.abs()
        sx, sy = torch.where(dx > 0, 1, -1).int(), torch.where(dy > 0, 1, -1).int()
        e, kx, ky = ax - ay, torch.zeros_like(hx), torch.zeros_like(hx)
        flat = out[lo:lo + n].view(-1)
        step = 0
        while idx.numel():
            xs = e >= 0
            kx += xs.int()
            ky += (~xs).int()
            e += torch.where(xs, -2 * ay, 2 * ax)
            cx, cy = hx + sx * kx, hy + sy * ky
            c2 = kx.long() * kx + ky.long() * ky
            live = (cx >= 0) & (cy >= 0) & (cx < w) & (cy < h) & (c2 <= lim)
            hit = live & occ[(cy.clamp(0, h - 1).long() * w + cx.clamp(0, w - 1).long())]
            r = torch.floor(torch.sqrt(c2[hit].double()) * 65536.0).long()
            r -= (r * r > c2[hit] << 32).long()
            r += ((r + 1) * (r + 1) <= c2[hit] << 32).long()
            flat[idx[hit]] = r
            live &= ~hit
            step += 1
            if step % 8 == 0:
                idx, hx, hy, ax, ay, sx, sy, e, kx, ky = (v[live] for v in (idx, hx, hy, ax, ay, sx, sy, e, kx, ky))
            else:   # rays that have ended stay where they cannot hit
                hx = torch.where(live, hx, torch.full_like(hx, -(1 << 28)))
    return out


def field_of(gt, C):
    """min(d^2, C) per cell, int32, with a border that reads C."""
    h, w = gt.shape
    r = math.isqrt(C)
    inf = 1 << 20
    occ = torch.nn.functional.pad(gt >= 65, (r, r, r, r))
    col = torch.full((h, w + 2 * r), inf, dtype=torch.int32, device="cuda")
    for dy in range(-r, r + 1):
        col = torch.where(occ[r + dy:r + dy + h], col.clamp(max=dy * dy), col)
    d2 = torch.full((h, w), C, dtype=torch.int32, device="cuda")
    for dx in range(-r, r + 1):
        d2 = torch.minimum(d2, col[:, r + dx:r + dx + w] + dx * dx)
    return d2


def survivors_of(case, gt, cells, b, R, iv_len):
    """Hypothesis indices in rank order."""
    ns, n = case["ns"], case["beams"]
    m = torch.arange(0, ns, ns // case["orient"], device="cuda")
    if n / ns >= 0.9:
        m = m[:1]
    scans = cast_sums(gt, cells, ns, case["max_range"])
    if case["coarse"] == "caer":
        num = torch.full((len(cells),), 1 << 60, dtype=torch.int64, device="cuda")
        for q in m.tolist():
            num = torch.minimum(num, (scans[:, (b + q) % ns] - R).abs().sum(1))
    else:
        P = torch.cat([torch.zeros((len(cells), 1), dtype=torch.int64, device="cuda"), torch.cat([scans, scans], 1).cumsum(1)], 1)
        s = (int(b[0]) + m) % ns
        num = (R.sum() - (P[:, s + iv_len] - P[:, s])).abs().amin(1)
    return num, torch.sort(num, stable=True).indices[:min(case["topk"], len(cells))]


def scores_of(case, gt, cells, surv, b, R):
    """float64 [K, orient]: the score of every survivor and orientation."""
    h, w = gt.shape
    ns = case["ns"]
    C = round(D_MAX / RES) ** 2
    field = field_of(gt, C).reshape(-1)
    valid = R > 0
    b, R = b[valid], R[valid]
    N = len(R)
    lam = case["beams"] / ns
    km = max(1, math.floor((0.9 + lam * (0.8 - 0.9)) * N))
    kl = max(1, math.floor((0.8 + lam * (0.6 - 0.8)) * N))
    k = sorted((N, km, kl))[1]
    v = torch.arange(C + 1, device="cuda", dtype=torch.float64)
    like = torch.log(torch.exp(-RES * RES * v / (2 * 0.2 ** 2)) + 1e-6)
    root = torch.sqrt(v)
    D = directions(ns)
    out = torch.empty((len(surv), case["orient"]), dtype=torch.float64, device="cuda")
    hc = to_gpu(cells).long()[surv]
    group = max(1, (1 << 26) // (N * len(surv)))
    for q0 in range(0, case["orient"], group):
        q = torch.arange(q0, min(q0 + group, case["orient"]), device="cuda")
        d = D[(b + q[:, None] * (ns // case["orient"])) % ns]
        o = (R[None, :, None] * d + (1 << 45)) >> 46
        x, y = hc[:, 0, None, None] + o[..., 0], hc[:, 1, None, None] + o[..., 1]
        inside = (x >= 0) & (y >= 0) & (x < w) & (y < h)
        e = torch.where(inside, field[y.clamp(0, h - 1) * w + x.clamp(0, w - 1)], C).to(torch.int16)
        e = torch.sort(e, -1).values.long()
        wp = torch.exp(like[e[..., :k]].mean(-1))
        dbar = RES * root[e].mean(-1)
        sd = (D_MAX - dbar).clamp(max=D_MAX - RES / 2) / (D_MAX - RES / 2)
        var = (RES * RES * e.double().mean(-1) - dbar * dbar).clamp(min=0)
        out[:, q0:q0 + len(q)] = (wp * sd.clamp(min=0) * torch.exp(-var / 2)).pow(1.0 / 3.0)
    return out


def exact(case, seed):
    if case["kind"] == "batch":   # the scores that run() returns are the first request's
        maps, reqs = batch_inputs(case, seed)
        (g, gt, cells), (_, z, angles, max_range, topk) = maps[0], reqs[0]
        ns = round(2.0 * math.pi / float(np.diff(angles.astype(np.float64))[:2].max()))
        case = {"beams": len(z), "ns": ns, "orient": case["orient"], "topk": topk, "max_range": max_range,
                "coarse": "smad", "early": False, "kind": "batch"}
    elif case["kind"] != "locate" or case["icp"]:
        return None   # whole numbers, or poses that follow from them (a refined pose ends the loop where its scores say)
    else:
        g, gt, cells, angles, z = inputs(case, seed)
    n, ns = case["beams"], case["ns"]
    b = to_gpu((np.arange(n) - n // 2) % ns)
    zd = z.astype(np.float64)
    ok = np.isfinite(zd) & (zd > 0) & (z < np.float32(case["max_range"]))
    R = to_gpu(np.where(ok, np.rint(zd * 65536.0 / RES), 0).astype(np.int64))
    num, surv = survivors_of(case, gt, cells, b, R, n)
    T = scores_of(case, gt, cells, surv, b, R)
    if case["early"]:
        for lo in range(0, len(surv), BATCH):
            if float(T[lo:lo + BATCH].max()) >= TAU:
                T[lo + BATCH:] = math.nan
                break
    if case["kind"] == "batch":
        return {"whole": None, "pose": None, "tam": None, "scores": T}
    out = dict.fromkeys(WHOLE + ("x", "y", "theta", "smad"))
    out.update(tam=float(torch.where(T.isnan(), torch.zeros_like(T), T).max()), scores=T, numerators=num)
    return out
