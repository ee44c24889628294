"""Kernels at the sizes where their tiling changes: remainders of tiles and
stages, the smallest and the largest of a range, both sides of a dispatch."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import full_case, relo, run, small_case, stages   # noqa: F401  (relo: the module fixture)

pytestmark = pytest.mark.gpu
RES = 0.05


@pytest.mark.parametrize("early", [False, True])
@pytest.mark.parametrize("n_orient", [6, 120])
@pytest.mark.parametrize("K", [1, 5, 17, 30])
def test_tam_tasks_of_few_survivors(relo, K, n_orient, early):
    """TAM tasks that split by orientation and tasks that do not, blocks of 4 and a remainder of 2 orientations: scores,
    argmax and survivors against the oracle (full_case's bounds)."""
    wl = small_case(n_orient=n_orient)
    full_case(relo, wl, K, early_stop=early, batch=7, local_topk=2, tau=2.0)[0].close()


@pytest.mark.parametrize("d_max_cells", [40, 80, 90])
def test_tam_tables_of_different_resolutions_in_one_batch(relo, d_max_cells):
    """Maps of different resolution have different likelihood tables: one launch scores both (a table per stage, and at
    the largest clamp a single stage), every result and the first request's scores as alone, bit for bit."""
    import torch
    wl = small_case()
    ctx = relo.Relo(n_orient=40, topk=30, batch=11, local_topk=3, early_stop=0, d_max=0.05 * d_max_cells)
    reqs = []
    for res in (0.05, 0.1, 0.05):
        mid = ctx.load_map(wl.grid, res)
        ctx.set_hypotheses(mid, workloads.cell_centres(wl.hyps, res))
        reqs.append((mid, wl.ranges * (res / 0.05), wl.angles, wl.max_range * (res / 0.05)))

    def scores(rows):
        return ctx.stage(relo.STAGE_TAM, torch.empty((rows, 40), device="cuda")).cpu().numpy()
    alone = []
    for q in reqs:
        alone.append((ctx.relocalize(*q).as_dict(), scores(30)))
    for first in range(3):
        order = [reqs[(first + i) % 3] for i in range(3)]
        got = ctx.relocalize_batch(order)
        assert [g.as_dict() for g in got] == [alone[(first + i) % 3][0] for i in range(3)]
        assert np.array_equal(scores(30).view(np.uint32), alone[first][1].view(np.uint32))
    ctx.close()


@pytest.mark.parametrize("cells,ns", [(1, 360), (33, 90), (7, 361)])
def test_synth_scans_beyond_the_32_bit_root(relo, cells, ns):
    """Hits on both sides of 1024 cells (where the range's square root changes form), against cell-by-cell stepping and
    the oracle."""
    import torch
    g = np.zeros((40, 1500), np.int8)
    g[0] = g[-1] = 100
    g[:, 0] = g[:, -1] = 100
    g[10:14, 1100] = 100
    xy = np.array([[3 + 2 * i, 20] for i in range(cells)], np.int32)
    ang = workloads.beam_angles(ns, ns)
    out = []
    for tables in (1, 0):
        ctx = relo.Relo(n_orient=0, ray_tables=tables)
        mid = ctx.load_map(g, RES)
        r, h = ctx.synth_scans(mid, torch.from_numpy(xy).cuda(), ang, 80.0, ns)
        out.append((r.cpu().numpy(), h.cpu().numpy()))
        ctx.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    pl = oracle.plan(np.full(ns, 1.0, np.float32), ang, 80.0, RES, oracle.Params(n_orient=0))
    for k in range(cells):
        want, hx, hy = oracle.synth_scan(g, int(xy[k, 0]), int(xy[k, 1]), pl)
        assert np.array_equal(out[0][0][k].astype(np.int64), want)
    assert (out[0][0] >= 1024 << 16).any() and (out[0][0] < 1024 << 16).any()


@pytest.mark.parametrize("rho,points", [(0.25, 164), (0.2, 256), (0.1998, 257), (0.14, 523)])
def test_rrt_sub_batches(relo, rho, points):
    """A round shorter than a sub-batch, exactly one, one point more, and two with a remainder: the serial tree, bit for
    bit, over several rounds."""
    import math

    import torch
    from rrt_f32 import serial_rrt
    g = workloads.make_room(1000)
    assert math.ceil(g.size * RES * RES / (rho * rho)) == points
    clr = workloads.clearance_table(g, RES)
    p0 = workloads.free_start(g, RES, 0.21, 7, clr)
    want, rounds, nodes = serial_rrt(clr, RES, p0, rho, 0.6, 0.21, 0, 5, max_rounds=6)
    ctx = relo.Relo()
    got, r, n = ctx.rrt_hypotheses(torch.tensor(clr, device="cuda"), RES, p0, rho, 0.6, 0.21, 0, seed=5, max_rounds=6)
    ctx.close()
    assert (r, n) == (rounds, nodes)
    assert np.array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("max_range", [30.0, 29.95, 30.3])   # border widths 601, 600 and 607: band phases 1, 0 and 7
@pytest.mark.parametrize("shape,density", [
    ((1, 1), 0.0), ((1, 1), 1.0), ((7, 300), 0.02), ((9, 1025), 0.001), ((65, 8), 0.05), ((64, 257), 0.01),
    ((129, 1024), 0.3), ((73, 1030), 0.0001),
    ((400, 700), -1.0),    # one occupied cell: distances beyond 16 bits, in both directions
    ((330, 515), -2.0),    # an occupied column at each end: far cells in the middle only
    ((40, 620), 0.0),      # none
])
def test_edt_bands(relo, shape, density, max_range):
    """Squared distances, likelihood field and occupancy from packed 16-bit bands and from the 32-bit pass, with sides and
    bands that do not divide, against the oracle; the allocation-free entry point where it applies."""
    import torch
    rng = np.random.default_rng(3)
    H, W = shape
    g = np.zeros(shape, np.int8)
    if density == -1.0:
        g[H // 3, W // 4] = 100
    elif density == -2.0:
        g[:, 0] = g[:, -1] = 65
    else:
        g[rng.random(shape) < density] = 100
        g[rng.random(shape) < 0.1] -= 1   # unknown cells, and occupied ones of other values
    want = oracle.edt(g)
    occ = g >= 65
    ctx = relo.Relo(max_range=max_range)
    gt = torch.from_numpy(g).cuda()
    for mid in (ctx.load_map(np.zeros_like(g), RES), ctx.load_map_dev(gt, RES)):
        ctx.update_map_dev(mid, gt)
        d2, field, o = (t.cpu().numpy() for t in ctx.map_tables(mid, g.shape))
        assert np.array_equal(d2, want)
        assert np.array_equal(field, np.where((want < 0) | (want > 1600), 1600, want))
        assert np.array_equal(o, occ)
    ctx.close()
    if max(shape) <= 1024:
        out = torch.full(shape, 7, dtype=torch.int32, device="cuda")
        odd = torch.empty(H * W + 1, dtype=torch.int8, device="cuda")   # a grid at an odd address
        odd[1:] = gt.reshape(-1)
        for ptr in (gt.data_ptr(), odd.data_ptr() + 1):
            out.fill_(7)
            assert relo.lib().relo_edt_noalloc(ptr, W, H, out.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
            assert np.array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("n_beams,ns,n_orient,gap", [
    (90, 120, 120, 0),     # every direction an orientation
    (90, 120, 40, 7),      # two intervals, three residue classes
    (100, 120, 2, 0),      # fewer orientations than a lane holds: lanes split the beams
    (300, 500, 500, 11),   # more orientations than one pass of a warp
    (31, 32, 16, 0),       # one beam short of the circle
])
def test_caer_orientation_groups(relo, n_beams, ns, n_orient, gap):
    """CAER numerators, shifts and survivors equal the oracle's across group, class and interval remainders."""
    wl = small_case(n_beams=n_beams, ns=ns, n_orient=n_orient)
    keep = np.ones(n_beams, bool)
    keep[n_beams // 3:n_beams // 3 + gap] = False
    wl.ranges, wl.angles = wl.ranges[keep].copy(), wl.angles[keep]
    wl.ranges[::9] = 100.0   # invalid beams
    full_case(relo, wl, 12, batch=5, local_topk=2, coarse=1)[0].close()


def test_caer_ranges_beyond_a_block_of_32_bits(relo):
    """A coarse map resolution makes the range limit 8000 cells: sums of differences leave 32 bits within a block."""
    g = np.zeros((30, 9000), np.int8)
    g[0] = g[-1] = 100
    g[:, 0] = g[:, -1] = 100
    hyps = np.array([[x, 15] for x in range(500, 1000, 100)], np.int32)
    ang = workloads.beam_angles(40, 60)
    z = np.random.default_rng(1).uniform(1.0, 399.0, 40).astype(np.float32)   # far from every synthesized range
    prm = dict(n_orient=60, topk=3, coarse=1)
    ctx = relo.Relo(n_orient=60, topk=3, coarse_metric=1, max_range=400.0, ray_tables=0)
    mid = ctx.load_map(g, RES)
    ctx.set_hypotheses(mid, workloads.cell_centres(hyps, RES))
    ctx.relocalize(mid, z, ang, 400.0)
    import torch
    got = ctx.stage(relo.STAGE_SMAD_NUM, torch.empty(len(hyps), dtype=torch.int64, device="cuda")).cpu().numpy()
    ctx.close()
    pl = oracle.plan(z, ang, 400.0, RES, oracle.Params(**prm))
    want, _ = oracle.coarse(g, hyps, pl, oracle.Params(**prm))
    assert np.array_equal(got, want) and want.max() > 1 << 32


@pytest.mark.parametrize("requests", [2, 5, 11, 24])
def test_icp_cluster_sizes(relo, requests):
    """8, 4, 2 and 1 CTAs per refined pose: each request of a batch gets the pose it gets alone (its sums are added in
    another order: 1e-9 m and rad, far above that and far below a cell) and its score (the same endpoints: equal)."""
    g = workloads.make_room(2, n=40, n_boxes=4)
    free = np.argwhere(g == 0)[:, ::-1]
    hyps = free[np.random.default_rng(2).choice(len(free), 60, replace=False)].astype(np.int32)
    ctx = relo.Relo(n_orient=40, topk=48, batch=16, local_topk=12, early_stop=0, icp_iters=10)
    mid = ctx.load_map(g, RES)
    ctx.set_hypotheses(mid, workloads.cell_centres(hyps, RES))
    reqs = []
    for i in range(requests):
        n = 60 + 5 * i
        ang = workloads.beam_angles(n, 120 if n <= 120 else 240)
        true = ((hyps[i][0] + 0.8) * RES, (hyps[i][1] + 0.3) * RES, 0.5 * i)
        z = workloads.render_scan(g, RES, true, ang, 6.0)
        reqs.append((mid, workloads.add_noise(z, 6.0, i, sigma=0.005, drop_frac=0.0, short_frac=0.0), ang, 6.0))
    alone = [ctx.relocalize(*q) for q in reqs]
    for a, b in zip(alone, ctx.relocalize_batch(reqs)):
        assert (a.hyp, a.m, a.n_batches, a.smad_num) == (b.hyp, b.m, b.n_batches, b.smad_num)
        assert abs(a.x - b.x) <= 1e-9 and abs(a.y - b.y) <= 1e-9
        assert abs((a.theta - b.theta + np.pi) % (2 * np.pi) - np.pi) <= 1e-9
        assert a.tam == b.tam
    ctx.close()


@pytest.mark.parametrize("shape,kind", [((700, 700), "free"), ((333, 1017), "sparse"), ((1017, 333), "sparse"),
                                        ((264, 2050), "corridor"), ((2050, 264), "corridor")])
def test_walk_boxes_of_every_slope(relo, shape, kind):
    """Rays of every slope class across boxes of up to 16 x 16 tiles, long and flat, tall and narrow, in maps whose sides
    are not multiples of 8: ranges and hit cells as cell-by-cell stepping gives them."""
    import torch
    rng = np.random.default_rng(11)
    H, W = shape
    g = np.zeros(shape, np.int8)
    if kind == "sparse":
        g[rng.random(shape) < 0.0002] = 100
    elif kind == "corridor":
        g[::89] = 100
        g[:, ::97] = 100
        g[rng.integers(0, H, 400), rng.integers(0, W, 400)] = 0
        for _ in range(40):
            y, x = int(rng.integers(0, H - 20)), int(rng.integers(0, W - 20))
            g[y:y + 20, x:x + 20] = 0
    free = np.argwhere(g == 0)[:, ::-1]
    cells = free[rng.choice(len(free), 60, replace=False)].astype(np.int32)
    ang = workloads.beam_angles(720, 720)
    out = []
    for tables in (1, 0):
        ctx = relo.Relo(n_orient=0, ray_tables=tables)
        mid = ctx.load_map(g, RES)
        r, h = ctx.synth_scans(mid, torch.from_numpy(cells).cuda(), ang, 60.0, 720)
        out.append((r.cpu().numpy(), h.cpu().numpy()))
        ctx.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("n_beams,ns,n_orient", [
    (20, 32, 8), (70, 128, 16), (71, 132, 33), (100, 160, 40), (500, 768, 96), (520, 772, 193), (90, 130, 65), (61, 97, 97),
])
def test_smad_row_blocks(relo, n_beams, ns, n_orient):
    """SMAD rows of less than a block, whole blocks and remainders, rows that are not 16-byte aligned, and gapped scans:
    numerators, shifts and survivors equal the oracle's."""
    wl = small_case(n_beams=n_beams, ns=ns, n_orient=n_orient)
    full_case(relo, wl, 12, batch=5, local_topk=2)[0].close()
    keep = np.ones(n_beams, bool)
    keep[n_beams // 2:n_beams // 2 + 5] = False
    wl.ranges, wl.angles = wl.ranges[keep].copy(), wl.angles[keep]
    full_case(relo, wl, 12, batch=5, local_topk=2)[0].close()


@pytest.mark.parametrize("ns,gap", [(64, 3), (130, 0), (131, 7), (720, 30), (721, 0)])
def test_smad_single_orientation_rows(relo, ns, gap):
    """Scans of 0.9 of the circle and more (m = 0 only): the row sums over aligned and unaligned intervals that may wrap."""
    wl = small_case(n_beams=ns, ns=ns, n_orient=1 if ns in (131, 721) else 2)
    for first in (0, ns // 3):   # the gap inside the scan, or the scan starting after it
        keep = np.ones(ns, bool)
        keep[first:first + gap] = False
        z, a = wl.ranges.copy(), wl.angles
        w = workloads.Workload("row", wl.grid, wl.res, wl.hyps, z[keep], a[keep], wl.max_range, wl.n_orient, 8, ns, (0, 0, 0))
        full_case(relo, w, 12, batch=5, local_topk=2)[0].close()


@pytest.mark.parametrize("copies,K", [(1, 30), (40, 700), (128, 30), (140, 700), (140, 1023), (600, 700), (200, 5), (700, 700),
                                      (700, 5)])
def test_topk_digits(relo, copies, K):
    """Hypotheses repeated so that many keys share a leading digit (ranks counted in short digits, long digits sorted,
    more keys of the last digit than are sorted; keys held in registers and not): survivors equal the oracle's ranking of the same numerators."""
    wl = small_case()
    hyps = np.repeat(wl.hyps, copies, axis=0)
    ctx, _, got = run(relo, wl.grid, wl.res, hyps, wl.ranges, wl.angles, wl.max_range, n_orient=wl.n_orient, topk=K,
                      batch=256, local_topk=2, early_stop=0)
    nb = -(-K // min(256, K))
    st = stages(relo, ctx, len(hyps), K, wl.n_orient, nb, 2)
    assert got.status == 0 and np.array_equal(st["surv"], oracle.rank(st["num"], K))
    ctx.close()


@pytest.mark.parametrize("n_orient", [305, 610, 1220])
def test_offsets_of_several_orientations_per_task(relo, n_orient):
    """Endpoint tables by blocks of 2, 4 and 8 orientations with a remainder: scores against the oracle (full_case)."""
    full_case(relo, small_case(n_beams=70, ns=1220, n_orient=n_orient), 3, batch=3, local_topk=2)[0].close()


@pytest.mark.parametrize("K,batch", [(30, 1), (700, 200), (1024, 16), (1300, 300), (2100, 1024)])
def test_select_batches_ranked_together(relo, K, batch):
    """Local top-k lists of many small batches, of a short last one, and of more positions than are ranked at once: the
    order of each batch's best scores (ties to the earlier survivor), and the best of all batches."""
    wl = small_case()
    hyps = np.repeat(wl.hyps, 70, axis=0)
    L = min(20, batch)
    ctx, _, got = run(relo, wl.grid, wl.res, hyps, wl.ranges, wl.angles, wl.max_range, n_orient=wl.n_orient, topk=K,
                      batch=batch, local_topk=L, early_stop=0)
    nb = -(-K // batch)
    st = stages(relo, ctx, len(hyps), K, wl.n_orient, nb, L)
    best = st["T"].max(axis=1)
    for b in range(nb):
        mine = best[b * batch:(b + 1) * batch]
        want = np.full(L, -1)
        order = np.argsort(-mine, kind="stable")[:L] + b * batch
        want[:len(order)] = order
        assert np.array_equal(st["local"][b], want)
    top = int(np.argmax(best))
    assert got.status == 0 and got.n_batches == nb and got.n_tam_evals == K * wl.n_orient
    assert got.hyp == st["surv"][top] and got.tam == best[top]
    ctx.close()


@pytest.mark.parametrize("shape,at", [
    ((30, 1300), (0, 0)),      # rows of 8 whose far cells fill the list of the 32-bit pass once and more
    ((41, 2100), (20, 1050)),  # on both sides of the occupied cell
    ((20, 8300), (3, 4)),      # wider than 8192: 4 rows at a time, several lists
])
def test_edt_lists_of_far_cells(relo, shape, at):
    """Bands with more groups of far cells than one list of the 32-bit pass holds, several times over: the oracle's
    distances and field in every update."""
    import torch
    g = np.zeros(shape, np.int8)
    g[at] = 100
    want = oracle.edt(g)
    ctx = relo.Relo(max_range=5.0)
    gt = torch.from_numpy(g).cuda()
    mid = ctx.load_map_dev(gt, RES)
    for _ in range(8):
        d2, field, _ = (t.cpu().numpy() for t in ctx.map_tables(mid, shape))
        assert np.array_equal(d2, want)
        assert np.array_equal(field, np.minimum(want, 1600))
        ctx.update_map_dev(mid, gt)
    ctx.close()


@pytest.mark.parametrize("shape", [(1, 4), (9, 256), (70, 300), (33, 1024)])   # rows of a multiple of 4 cells
def test_edt_noalloc_output_at_any_int(relo, shape):
    """An output that starts at any int32 of a buffer (a part of the caller's own pool), with a guard on both sides."""
    import torch
    H, W = shape
    g = np.zeros(shape, np.int8)
    g[np.random.default_rng(4).random(shape) < 0.01] = 100
    g[0, 0] = 100
    want = oracle.edt(g)
    gt = torch.from_numpy(g).cuda()
    for first in (4, 5, 6, 7):   # 0 to 3 ints past a 16-byte boundary
        pool = torch.full((H * W + 12,), 7, dtype=torch.int32, device="cuda")
        assert pool.data_ptr() % 16 == 0
        assert relo.lib().relo_edt_noalloc(gt.data_ptr(), W, H, pool.data_ptr() + 4 * first,
                                           torch.cuda.current_stream().cuda_stream) == 0
        got = pool.cpu().numpy()
        assert np.array_equal(got[first:first + H * W].reshape(shape), want)
        assert (got[:first] == 7).all() and (got[first + H * W:] == 7).all()


def load_widths(widths):
    """Maps of these widths in this order: tables equal to the oracle's."""
    import paper_2511_01219_gb300 as relo
    for W in widths:
        g = np.zeros((21, W), np.int8)
        g[np.random.default_rng(W).random(g.shape) < 0.005] = 100
        g[:, W // 2 - 200:W // 2 + 200] = 0   # far cells in the middle
        want = oracle.edt(g)
        ctx = relo.Relo(max_range=5.0)
        mid = ctx.load_map(g, RES)
        d2, field, _ = (t.cpu().numpy() for t in ctx.map_tables(mid, g.shape))
        ctx.close()
        assert np.array_equal(d2, want) and np.array_equal(field, np.minimum(want, 1600)), W


def test_map_widths_around_the_shared_memory_limits(relo):
    """Widths on both sides of the sizes at which the 32-bit pass asks for more shared memory than a kernel gets unasked,
    and takes 4 rows at a time; smallest first, in a process where no wider map has asked for more before."""
    here = os.path.dirname(os.path.abspath(__file__))
    code = "import test_gpu_kernel_edges as t; t.load_widths([2535, 2560, 2800, 3072, 3073, 8192, 8193])"
    subprocess.check_call([sys.executable, "-c", code], cwd=here,
                          env={**os.environ, "PYTHONPATH": os.pathsep.join([here, os.path.dirname(here)])}, timeout=300)


@pytest.mark.parametrize("order", ["sensors", "swapped", "late_start"])
@pytest.mark.parametrize("coarse", [0, 1])
def test_beams_out_of_cyclic_order(relo, coarse, order):
    """Scans whose beams are not listed in cyclic order but pass the grid's checks: three sensors one after the other, two
    neighbours swapped, and both with a first beam in the middle of an interval.  SMAD's and CAER's numerators, shifts and
    survivors equal the oracle's, which takes every beam by its own direction."""
    wl = small_case(n_beams=40, ns=40, n_orient=20)
    idx = {"sensors": [*range(10), *range(20, 30), *range(10, 20)],
           "swapped": [0, 1, 2, 4, 3, *range(5, 30)],
           "late_start": [*range(5, 12), *range(14, 30), 3, 4, 1, 2, 0]}[order]
    wl.ranges, wl.angles = wl.ranges[idx].copy(), wl.angles[idx].copy()
    wl.ranges[::7] = 100.0   # invalid beams
    full_case(relo, wl, 12, batch=5, local_topk=2, coarse=coarse)[0].close()


@pytest.mark.parametrize("n_beams,ns,n_orient", [(28, 32, 32), (50, 64, 16), (65, 97, 97), (300, 361, 361), (32, 32, 8),
                                                 (2048, 8192, 64)])
def test_smad_ranges_whose_chunks_pass_32_bits(relo, n_beams, ns, n_orient):
    """Ranges of some 2300 cells: 32 of them sum to more than 2^32 in Q16.  Numerators and shifts equal the oracle's by
    prefixes, by the window tables that a cached call builds, and when it reads them; a short-range request beside them."""
    import torch
    n = 4200
    g = np.zeros((n, n), np.int8)
    g[0] = g[-1] = 100
    g[:, 0] = g[:, -1] = 100
    hyps = np.array([[2100, 2100], [2060, 2130], [2155, 2045]], np.int32)
    ang = workloads.beam_angles(n_beams, ns)
    z = np.random.default_rng(ns).uniform(95.0, 145.0, n_beams).astype(np.float32)
    prm = oracle.Params(n_orient=n_orient, topk=2)
    pl = oracle.plan(z, ang, 150.0, RES, prm)
    row, _, _ = oracle.synth_scan(g, 2100, 2100, pl)
    assert int(row[:32].astype(np.int64).sum()) > 1 << 32
    want, shift = oracle.coarse(g, hyps, pl, prm)
    near = workloads.make_room(3, n=40, n_boxes=4)
    near_hyps = np.argwhere(near == 0)[:3, ::-1].astype(np.int32)
    near_z = np.where(z > 120.0, 1.0, 0.5).astype(np.float32)
    near_want, _ = oracle.coarse(near, near_hyps, oracle.plan(near_z, ang, 4.0, RES, prm), prm)

    def numerators(ctx):
        k = len(hyps)
        return (ctx.stage(relo.STAGE_SMAD_NUM, torch.empty(k, dtype=torch.int64, device="cuda")).cpu().numpy(),
                ctx.stage(relo.STAGE_SMAD_M, torch.empty(k, dtype=torch.int32, device="cuda")).cpu().numpy())
    for cache, calls in ((0, 1), (1 << 30, 3)):
        ctx = relo.Relo(n_orient=n_orient, topk=2, early_stop=0, max_range=150.0, scan_cache_bytes=cache)
        far_map, near_map = ctx.load_map(g, RES), ctx.load_map(near, RES)
        ctx.set_hypotheses(far_map, workloads.cell_centres(hyps, RES))
        ctx.set_hypotheses(near_map, workloads.cell_centres(near_hyps, RES))
        for _ in range(calls):
            ctx.relocalize(far_map, z, ang, 150.0)
            num, m = numerators(ctx)
            assert np.array_equal(num, want) and np.array_equal(m, shift)
        ctx.relocalize_batch([(near_map, near_z, ang, 4.0), (far_map, z, ang, 150.0)])
        assert np.array_equal(numerators(ctx)[0], near_want)   # the first request's stages
        ctx.close()


def test_stages_end_with_the_scratch_they_lie_in(relo):
    """The stages of a served batch once the server has stopped, and those of a call whose scratch a later call, too large
    for the budget, has given up: an error, not a read of freed memory."""
    import torch
    wl = small_case()

    def stage_error(ctx):
        with pytest.raises(relo.ReloError) as e:
            ctx.scan_info()
        assert e.value.code == relo.E_NOT_FOUND
        with pytest.raises(relo.ReloError) as e:
            ctx.stage(relo.STAGE_SURVIVORS, torch.empty(64, dtype=torch.int32, device="cuda"))
        assert e.value.code == relo.E_NOT_FOUND
    ctx = relo.Relo(n_orient=40, topk=8)
    mid = ctx.load_map(wl.grid, RES)
    ctx.set_hypotheses(mid, workloads.cell_centres(wl.hyps, RES))
    ctx.serve_start(4, 2)
    t = ctx.submit(mid, wl.ranges, wl.angles, wl.max_range)
    while ctx.poll(t) is None:
        pass
    ctx.serve_stop()
    stage_error(ctx)
    ctx.relocalize(mid, wl.ranges, wl.angles, wl.max_range)
    assert ctx.scan_info()[0] == 120   # a call's own stages are there again
    ctx.close()
    many = np.repeat(wl.hyps, 1000, axis=0)
    ctx = relo.Relo(n_orient=40, topk=8, max_range=wl.max_range, hbm_budget=8 << 20)   # less than the rows below alone
    small = ctx.load_map(wl.grid, RES)
    ctx.set_hypotheses(small, workloads.cell_centres(wl.hyps, RES))
    large = ctx.load_map(wl.grid, RES)
    ctx.set_hypotheses(large, workloads.cell_centres(many, RES))
    ctx.relocalize(small, wl.ranges, wl.angles, wl.max_range)
    assert ctx.scan_info()[0] == 120
    with pytest.raises(relo.ReloError) as e:
        ctx.relocalize(large, wl.ranges, wl.angles, wl.max_range)   # 30000 rows of 120 ranges: 14 MB
    assert e.value.code == relo.E_OVER_BUDGET
    stage_error(ctx)
    ctx.close()


@pytest.mark.parametrize("scans", [33, 70])
def test_batch_of_more_scans_than_plans_are_kept(relo, scans):
    """A batch whose requests all have a beam grid of their own, more than the context keeps between calls: every result as
    alone, in the batch and in a second one."""
    wl = small_case(n_beams=110)
    ctx = relo.Relo(n_orient=40, topk=8, batch=4, local_topk=2)
    mid = ctx.load_map(wl.grid, RES)
    ctx.set_hypotheses(mid, workloads.cell_centres(wl.hyps, RES))
    reqs = [(mid, wl.ranges[:40 + i], wl.angles[:40 + i], wl.max_range) for i in range(scans)]
    alone = [ctx.relocalize(*q).as_dict() for q in reqs]
    for _ in range(2):
        assert [r.as_dict() for r in ctx.relocalize_batch(reqs)] == alone
    ctx.close()
