"""Sizes at which the tiled kernels can go wrong: partial batches, tiles and rows, ties, unaligned arrays (GPU)."""
import numpy as np
import pytest
import torch

import bench
import oracle
import synth
from paper_2509_12138_gb300 import Frame, Units
from paper_2509_12138_gb300 import init as gi
from tests.gpu_util import captured_kernels

pytestmark = pytest.mark.gpu


def _points(n, seed):
    pts, nrm, _ = synth.interface_points(n, 8, seed)
    p, m = torch.from_numpy(pts).cuda(), torch.from_numpy(nrm).cuda()
    return (p, m) + gi.knn(p, 16)


def _weights(seed):
    w = gi.init_weights(seed)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    w[7168 + 64 + 4096 + 64:-8] = 0.1 * torch.randn(512, generator=g, device="cuda")
    return w


def _off_by_one(t):
    """The same rows in storage that starts 4 bytes past a 16-byte boundary."""
    s = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    v = s[1:].view(t.shape)
    v.copy_(t)
    return v


@pytest.mark.parametrize("n", [1, 127, 128, 129, 300])
@pytest.mark.parametrize("aligned", [True, False])
def test_mlp_forward_partial_batches(n, aligned):
    """A point's outputs and features do not depend on the points behind it, nor on how its rows are aligned."""
    p, m, idx, dist = _points(700, 1)
    w = _weights(2)
    full, feat = gi.mlp_forward(w, p, m, idx, dist), gi.mlp_features(p, m, idx, dist)
    # neighbours may lie past the first n points: the point arrays stay whole, the rows end at n
    i, d = (idx[:n], dist[:n]) if aligned else (_off_by_one(idx[:n]), _off_by_one(dist[:n]))
    L = gi._lib.load()
    out = torch.empty((n, 8), device="cuda")
    gi.check(L.gs_mlp_forward(gi._ptr(p), gi._ptr(m), gi._ptr(i), gi._ptr(d), n, gi._ptr(w), gi._ptr(out),
                              gi._stream()), "gs_mlp_forward")
    x = torch.empty((n, 112), dtype=torch.int16, device="cuda")
    gi.check(L.gs_mlp_features(gi._ptr(p), gi._ptr(m), gi._ptr(i), gi._ptr(d), n, gi._ptr(x), gi._stream()),
             "gs_mlp_features")
    assert torch.equal(out, full[:n]) and torch.equal(x, feat[:n])


@pytest.mark.parametrize("n,aligned", [(1, True), (127, True), (129, False), (128 * 152 + 3, True)])
def test_mlp_train_partial_batches(n, aligned):
    """Gradients and loss of one step against torch in 64 bits.  Every GEMM operand is rounded to bf16 (2^-9
    relative each; activation, signal and weight along three layers), so a gradient of random-signed terms lies
    within a few 2^-9 of the 64-bit one in norm; 2^-6 leaves a factor of about 3.  A point left out or counted
    twice changes it by about n^-1/2 (the small sizes), a CTA's share by more."""
    p, m, idx, dist = _points(max(n, 200), 3)
    w, g = _weights(4), torch.Generator(device="cuda")
    g.manual_seed(n)
    t = 0.5 * torch.randn((n, 8), generator=g, device="cuda")
    i, d = (idx[:n], dist[:n]) if aligned else (_off_by_one(idx[:n]), _off_by_one(dist[:n]))
    tr = gi.MLPTrainer(w.clone())
    loss = float(tr.step(p, m, i, d, t, n=n))
    q = w.double().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = torch.split(q, [7168, 64, 4096, 64, 512, 8])
    P, N, J, D = p.double(), m.double(), idx[:n].long(), dist[:n].double()
    X = torch.cat([((P[J] - P[:n, None]) / D.mean(1)[:, None, None]).reshape(n, 48), N[J].reshape(n, 48), N[:n]], 1)
    h = torch.relu(X @ W1.reshape(112, 64)[:99] + b1)
    h = torch.relu(h @ W2.reshape(64, 64) + b2)
    ref = (h @ W3.reshape(64, 8) + b3 - t).square().sum() / (8 * n)
    ref.backward()
    err = ((tr.grad - q.grad).norm() / q.grad.norm()).item()
    print(f"n {n}: gradient error {err:.2e}, loss {loss:.6f} against {ref.item():.6f}")
    assert err <= 2.0 ** -6 and abs(loss - ref.item()) <= 2.0 ** -6 * ref.item()


@pytest.mark.parametrize("n,k", [(2, 3), (5, 8), (17, 16), (4096, 16), (4096, 8), (4096, 3)])
def test_knn_ties_exact(n, k):
    """Points of a small lattice, many of them repeated: squared distances are exact in float32 and tie in large
    groups, so the neighbours are exactly the first k by (distance, index)."""
    g = np.random.default_rng(n + k)
    pts = (g.integers(0, 9, (n, 3)) / 8.0).astype(np.float32)
    idx, dist = (a.cpu().numpy() for a in gi.knn(torch.from_numpy(pts).cuda(), k))
    q = (pts * 8).astype(np.int64)
    for i in range(0, n, max(1, n // 200)):
        d2 = ((q - q[i]) ** 2).sum(1)
        o = np.lexsort((np.arange(n), d2))
        o = o[o != i][:k]
        want = np.full(k, -1)
        want[:len(o)] = o
        wd = np.full(k, np.inf, np.float32)
        wd[:len(o)] = np.sqrt((d2[o] / 64.0).astype(np.float32))
        assert np.array_equal(idx[i], want) and np.array_equal(dist[i], wd)


def _knn_on_grid(pts, k, lo, h, dims, aligned=True):
    """gs_knn on a grid of the caller's choice; aligned False: results to arrays 4 bytes past a 16-byte boundary."""
    L, n = gi._lib.load(), len(pts)
    p = torch.from_numpy(pts).cuda()
    lo, dims = np.asarray(lo, np.float32), np.asarray(dims, np.int32)
    dp = dims.ctypes.data_as(gi._lib.c_i32p)
    ws = torch.empty(L.gs_knn_workspace_size(n, dp), dtype=torch.uint8, device="cuda")
    idx, dist = torch.empty((n, k), dtype=torch.int32, device="cuda"), torch.empty((n, k), device="cuda")
    if not aligned:
        idx, dist = _off_by_one(idx), _off_by_one(dist)
    gi.check(L.gs_knn(gi._ptr(p), n, k, lo.ctypes.data_as(gi._lib.c_f32p), h, dp, gi._ptr(ws), ws.numel(),
                      gi._ptr(idx), gi._ptr(dist), gi._stream()), "gs_knn")
    return idx.cpu().numpy(), dist.cpu().numpy()


def _nearest_on_lattice(pts, i, k):
    """The k nearest others of point i by (distance, index), exact for points on a lattice of eighths."""
    q = (pts * 8).astype(np.int64)
    d2 = ((q - q[i]) ** 2).sum(1)
    o = np.lexsort((np.arange(len(pts)), d2))
    o = o[o != i][:k]
    return o, np.sqrt((d2[o] / 64.0).astype(np.float32))


@pytest.mark.parametrize("k", [3, 8, 16])
@pytest.mark.parametrize("cells", [1, 2, 8])
def test_knn_points_outside_the_grid(k, cells):
    """Points from outside the grid are held by its outermost cells and have the neighbours that all points' distances
    give, whichever side of it they and their neighbours lie on."""
    g = np.random.default_rng(k + cells)
    pts = (g.integers(-12, 21, (700, 3)) / 8.0).astype(np.float32)
    pts[:20] += 40.0  # a group far away from the grid
    idx, dist = _knn_on_grid(pts, k, (0.0, 0.0, 0.0), 1.0 / cells, (cells,) * 3)
    for i in range(len(pts)):
        want, wd = _nearest_on_lattice(pts, i, k)
        assert np.array_equal(idx[i], want) and np.array_equal(dist[i], wd)


@pytest.mark.parametrize("k", [3, 8, 16])
def test_knn_distances_past_the_float_range(k):
    """A point whose squared distance overflows float32 is no neighbour: its slot is -1 / inf, as with too few points."""
    x = np.array([0.0, 1.0, 2.0, 1e20, 1e20 + 1e13, 3e20, np.nan, np.inf], np.float32)
    pts = np.zeros((len(x), 3), np.float32)
    pts[:, 0] = x
    idx, dist = _knn_on_grid(pts, k, (-1.0, -1.0, -1.0), 1e20, (4, 1, 1))
    with np.errstate(over="ignore", invalid="ignore"):
        d2 = (x[:, None] - x[None, :]) ** 2
    for i in range(len(x)):
        near = sorted((d2[i, j], j) for j in range(len(x)) if j != i and np.isfinite(d2[i, j]))[:k]
        assert idx[i].tolist() == [j for _, j in near] + [-1] * (k - len(near))
        assert dist[i].tolist() == [float(np.sqrt(d)) for d, _ in near] + [np.inf] * (k - len(near))


@pytest.mark.parametrize("n,k", [(5, 8), (17, 16), (600, 16), (600, 8)])
def test_knn_unaligned_results(n, k):
    """Rows of results that do not start on 16 bytes are stored one value at a time: the same indices and distances."""
    pts = np.random.default_rng(n + k).uniform(0, 1, (n, 3)).astype(np.float32)
    want, got = (_knn_on_grid(pts, k, (-0.1, -0.1, -0.1), 0.25, (5, 5, 5), aligned) for aligned in (True, False))
    assert np.array_equal(want[0], got[0]) and np.array_equal(want[1], got[1])


@pytest.mark.parametrize("W,H,units", [(1, 1, 1), (31, 33, 2), (32, 32, 1), (65, 10, 3), (100, 71, 2)])
def test_loss_partial_tiles(W, H, units):
    """Image edges inside the loss kernels' tiles, planes that are no multiple of 16 bytes, several units; bounds
    as for the larger images: 1e-5 of the loss, 1e-3 of the largest gradient."""
    g = np.random.default_rng(W * H)
    img, gt = (g.uniform(0, 1, (units, 3, H, W)).astype(np.float32) for _ in range(2))
    mask = (g.uniform(0, 1, (units, H, W)) < 0.6).astype(np.uint8)
    mask[:, 0, 0] = 1
    fr = Frame(1, Units.single(1, units), W, H, 0, with_backward=False)
    fr.img.copy_(torch.from_numpy(img))
    loss = float(fr.loss(torch.from_numpy(gt).cuda(), torch.from_numpy(mask).cuda(), 0.2))
    ref = [oracle.loss(img[u].astype(np.float64), gt[u].astype(np.float64), mask[u], 0.2) for u in range(units)]
    assert loss == pytest.approx(np.mean([r[0] for r in ref]), rel=1e-5)
    d = np.stack([r[1] for r in ref]) / units
    assert np.abs(fr.dimg.cpu().numpy() - d).max() <= 1e-3 * np.abs(d).max()


@pytest.mark.parametrize("W,H,units", [(4, 1, 1), (32, 32, 1), (36, 45, 2), (100, 71, 2)])
def test_loss_unaligned_arrays(W, H, units):
    """Rows that start on 16 bytes are read 4 pixels at a time, others one by one: the same gradient, bit for bit; the
    mask has rows and columns with single pixels."""
    g = np.random.default_rng(W + H)
    gt = torch.from_numpy(g.uniform(0, 1, (units, 3, H, W)).astype(np.float32)).cuda()
    mask = torch.from_numpy((g.uniform(0, 1, (units, H, W)) < 0.3).astype(np.uint8)).cuda()
    mask[:, :, W // 2:] = 0
    mask[:, 0, 0] = 1
    fr = Frame(1, Units.single(1, units), W, H, 0, with_backward=False)
    fr.img.copy_(torch.from_numpy(g.uniform(0, 1, (units, 3, H, W)).astype(np.float32)))
    fr.loss(gt, mask, 0.2)
    want = fr.dimg.clone()
    assert float(want.abs().max()) > 0
    for a, b in ((_off_by_one(gt), mask), (gt, _off_by_one(mask)), (_off_by_one(gt), _off_by_one(mask))):
        fr.dimg.fill_(7.0)
        fr.loss(a, b, 0.2)
        assert torch.equal(fr.dimg, want)


def _lists_by_numpy(fr, cap):
    """The lists gs_bin_sort documents, from the projected records: instances in (depth, record index, tile) order,
    the first cap of them kept, each list in that order."""
    t = lambda a: a.cpu().numpy()  # noqa: E731
    P = fr.P
    tiles, depth, rad, xy = t(fr.tiles)[:P], t(fr.depth)[:P], t(fr.radius)[:P].astype(np.int64), fr.xy64()[:P]
    fu, fv = np.floor(xy[:, 0]).astype(np.int64), np.floor(xy[:, 1]).astype(np.int64)
    x0, x1 = (np.clip((fu + s) // 16, 0, fr.TX) for s in (-rad, rad + 15))
    y0, y1 = (np.clip((fv + s) // 16, 0, fr.TY) for s in (-rad, rad + 15))
    unit = np.searchsorted(fr.units.proj_base, np.arange(P), side="right") - 1
    lists = [[] for _ in range(fr.units.n * fr.n_tiles)]
    left = cap
    for p in np.lexsort((np.arange(P), depth.view(np.uint32))):
        if tiles[p] == 0:
            continue
        for ty in range(y0[p], y1[p]):
            for tx in range(x0[p], x1[p]):
                if left > 0:
                    lists[unit[p] * fr.n_tiles + ty * fr.TX + tx].append(p)
                    left -= 1
    return lists, cap - left


@pytest.mark.parametrize("n,views,W,H,cap", [
    (1, 1, 16, 16, 64), (33, 2, 40, 24, 1000), (1025, 3, 100, 60, 1 << 15), (1500, 2, 64, 64, 2000),
    (1500, 2, 64, 64, 1), (16384, 1, 48, 48, 1 << 17), (16385, 1, 48, 48, 1 << 17), (700, 1, 1024, 1024, 1 << 15),
    (300, 1, 1040, 1024, 1 << 15), (500, 1, 2048, 1024, 1 << 16), (500, 1, 2064, 1024, 1 << 16)])
def test_sort_lists_at_design_limits(n, views, W, H, cap):
    """Both sides of the small sort's limits (records per unit, number of lists), partial warps and rounds, several
    units, and a capacity that runs out, inside a record too: lists, ranges, counts and the chunk jobs."""
    g = synth.random_gaussians(n, 0, n + views, extent=0.8, log_scale_range=(-4.0, -2.0))
    cams = synth.orbital_cameras(8, 3.0, width=W, height=H).subset(list(range(views)))
    import paper_2509_12138_gb300 as gs
    fr = Frame(n, Units.single(n, views), W, H, 0, max_instances=cap, with_backward=False, with_loss=False, chunk=32)
    fr.preprocess(gs.pack_params(g, 0), gs.pack_cameras(cams))
    total = fr.total_instances()
    fr.sort()
    want, kept = _lists_by_numpy(fr, cap)
    assert fr.read_status() == (2 if total > cap else 0) and fr.instances() == kept == min(total, cap)
    vals, ranges = fr.sorted_lists()
    lens = ranges[:, 1] - ranges[:, 0]
    assert np.array_equal(lens, [len(w) for w in want])
    assert sorted(ranges[lens > 0, 0].tolist()) == np.cumsum([0] + [len(w) for w in want if w])[:-1].tolist()
    for (a, b), w in zip(ranges, want):
        assert vals[a:b].tolist() == w
    order, base = fr.tile_order.cpu().numpy(), fr.job_base.cpu().numpy()
    jobs = fr.jobs.cpu().numpy()[:2 * base[-1]].reshape(-1, 2)
    chunks = (lens[order] + 31) // 32
    assert sorted(order.tolist()) == list(range(len(lens))) and np.array_equal(np.diff(base), chunks)
    assert np.array_equal(jobs[:, 0], np.repeat(np.arange(len(order)), chunks))
    assert np.array_equal(jobs[:, 1], np.concatenate([np.arange(c) for c in chunks]))


@pytest.mark.parametrize("n,views,W,H,cap", [
    (3072, 1, 48, 48, 6144), (3073, 1, 48, 48, 6146), (4096, 3, 80, 64, 1 << 17), (16384, 1, 48, 48, 1 << 20),
    (5000, 2, 64, 64, 4097), (9000, 1, 200, 150, 13001), (9000, 2, 100, 60, 20000), (9000, 2, 100, 60, 1)])
def test_sort_lists_at_record_limit(n, views, W, H, cap):
    """Both sides of the small sort's limits of records per unit, and a capacity that runs out in the general design:
    in its first window of 4,096 staged instances, behind it, and inside a record."""
    test_sort_lists_at_design_limits(n, views, W, H, cap)


@pytest.mark.parametrize("n,views,W,H,cap,small", [
    (3072, 1, 48, 48, 2, True), (3073, 1, 48, 48, 2, False), (4096, 1, 64, 64, 4, True), (4097, 1, 64, 64, 4, False),
    (6144, 8, 128, 128, 4, True), (6145, 8, 128, 128, 4, False), (16384, 1, 64, 64, 4, False),
    (16384, 1, 64, 64, 52, True), (16384, 1, 64, 64, 51, False), (16385, 1, 64, 64, 60, False),
    (500, 1, 2048, 512, 4, True), (500, 1, 2048, 1024, 4, False)])
def test_sort_design_by_sizes(n, views, W, H, cap, small):
    """The small sort's four launches up to 4,096 lists and 1,024 log2(tiles) + 256 (capacity per record - 4) records
    per unit, at least 3,072 and at most 16,384; the general design's beyond, the faster one unless a splat is large."""
    import paper_2509_12138_gb300 as gs
    g = synth.random_gaussians(n, 0, n, extent=0.8, log_scale_range=(-4.0, -3.0))
    cams = synth.orbital_cameras(8, 3.0, width=W, height=H).subset(list(range(views)))
    fr = Frame(n, Units.single(n, views), W, H, 0, max_instances=cap * n * views, with_backward=False, with_loss=False)
    fr.preprocess(gs.pack_params(g, 0), gs.pack_cameras(cams))
    kernels = captured_kernels(fr.sort)
    assert kernels == 4 if small else kernels >= 18


@pytest.mark.parametrize("array", ["tiles", "depth"])
def test_sort_unaligned_records(array):
    """Records whose tile counts or depths do not start on 16 bytes are counted one at a time: the same lists."""
    import paper_2509_12138_gb300 as gs
    n = 3 * 2048 + 5
    g = synth.random_gaussians(n, 0, 6, extent=0.8, log_scale_range=(-5.0, -3.0))
    cams = gs.pack_cameras(synth.orbital_cameras(8, 3.0, width=1040, height=1040).subset([0]))
    fr = Frame(n, Units.single(n, 1), 1040, 1040, 0, with_backward=False, with_loss=False)
    fr.fit_capacity(gs.pack_params(g, 0), cams)
    fr.sort()
    want = fr.sorted_lists()
    moved = _off_by_one(getattr(fr, array))
    setattr(fr.proj, array, moved.data_ptr())
    fr.sorted_vals.zero_()
    fr.sort()
    got = fr.sorted_lists()
    assert fr.read_status() == 0 and len(want[0]) > n
    assert np.array_equal(want[0], got[0]) and np.array_equal(want[1], got[1])


@pytest.mark.parametrize("wide", [False, True])
def test_sort_of_many_records_equals_global(wide):
    """2^24 records on: with room for two instances a record the emission reads packed rectangles (wide: some are
    too wide to pack), with one less it reads the records; both give the global sort's lists, bit for bit."""
    import paper_2509_12138_gb300 as gs
    n = (1 << 24) + 77
    g = synth.random_gaussians(n, 0, 5, extent=0.9, log_scale_range=(-7.5, -6.0))
    if wide:
        g["log_scales"][::200_003] = -1.0
    cams = gs.pack_cameras(synth.orbital_cameras(8, 3.0, width=333, height=250).subset([1]))
    params = gs.pack_params(g, 0)
    del g
    got = []
    for cap, design in ((2 * n, "depth_first"), (2 * n - 1, "depth_first"), (2 * n, "global")):
        fr = Frame(n, Units.single(n, 1), 333, 250, 0, max_instances=cap, with_backward=False, with_loss=False)
        fr.preprocess(params, cams)
        fr.sort(design)
        count = fr.instances()
        assert fr.read_status() == 0 and 0 < count <= cap
        got.append([fr.sorted_vals[:count].cpu(), fr.ranges.cpu(), fr.block_masks[:count].cpu()])
        del fr
    for other in got[:2]:
        assert all(torch.equal(a, b) for a, b in zip(other, got[2]))


def _many_records(n, views, W, H, seed=5):
    """n splats of about a pixel (every 200,003rd one of many tiles) as parameters on the device, and their cameras."""
    import paper_2509_12138_gb300 as gs
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    params = torch.zeros((gs.param_planes(0), n, 4), device="cuda")
    params[0, :, :3] = 1.8 * torch.rand((n, 3), generator=g, device="cuda") - 0.9
    params[1, :, :3] = -6.5 + 0.5 * torch.randn((n, 3), generator=g, device="cuda")
    params[1, ::200_003, :3] = -1.0
    params[2] = torch.randn((n, 4), generator=g, device="cuda")
    return params, gs.pack_cameras(synth.orbital_cameras(8, 3.0, width=W, height=H).subset(list(range(views))))


@pytest.mark.parametrize("views,masks", [(1, True), (2, True), (1, False)])
def test_sort_by_packed_rectangles_equals_global(views, masks):
    """2^25 records on: with room for two instances a record the emission reads packed rectangles, with one less it
    reads the records; one view and several, with block masks and without: the global sort's lists, bit for bit."""
    n = (1 << 25) // views + 77
    params, cams = _many_records(n, views, 333, 250)
    got = []
    for cap, design in ((2 * views * n, "depth_first"), (2 * views * n - 1, "depth_first"), (2 * views * n, "global")):
        fr = Frame(n, Units.single(n, views), 333, 250, 0, max_instances=cap, with_backward=False, with_loss=False)
        fr.use_masks = masks
        fr.preprocess(params, cams)
        fr.sort(design)
        count = fr.instances()
        assert fr.read_status() == 0 and n * views // 2 < count <= cap
        got.append([fr.sorted_vals[:count].clone(), fr.ranges.clone()])
        if masks:
            got[-1].append(fr.block_masks[:count].clone())
        del fr
    for other in got[:2]:
        assert all(torch.equal(a, b) for a, b in zip(other, got[2]))


def test_sort_by_packed_rectangles_keeps_the_nearest():
    """More instances than the capacity behind packed rectangles: every list keeps its first entries, the capacity is
    full, and nothing dropped is nearer than anything kept."""
    n = (1 << 25) + 77
    params, cams = _many_records(n, 1, 1200, 900)
    params[1, :, :3] += 0.9  # some three instances a record
    out = []
    for cap in (4 * n, 2 * n):
        fr = Frame(n, Units.single(n, 1), 1200, 900, 0, max_instances=cap, with_backward=False, with_loss=False)
        fr.preprocess(params, cams)
        fr.sort()
        out.append((fr.read_status(), fr.instances(), fr.sorted_vals.clone(), fr.ranges.long().clone(), fr.depth.clone()))
        del fr
    (sa, na, va, ra, depth), (sb, nb, vb, rb, _) = out
    assert sa == 0 and sb == 2 and nb == 2 * n < na <= 4 * n
    la, lb = ra[:, 1] - ra[:, 0], rb[:, 1] - rb[:, 0]
    assert bool((lb <= la).all()) and int(lb.sum()) == nb
    list_of = torch.repeat_interleave(torch.arange(len(lb), device="cuda"), lb)
    within = torch.arange(nb, device="cuda") - rb[list_of, 0]
    assert torch.equal(vb[:nb], va[ra[list_of, 0] + within])
    cut = torch.ones(na, dtype=torch.bool, device="cuda")
    cut[ra[list_of, 0] + within] = False
    assert float(depth[vb[:nb].long()].max()) <= float(depth[va[:na][cut].long()].min())


@pytest.mark.parametrize("n,W,H,log_scales", [
    (3000, 100, 60, (-4.0, -2.5)),    # few short lists: no split
    (30000, 100, 60, (-3.5, -2.5)),   # fewer blocks than warps, long lists: everything behind the first chunk
    (60000, 500, 500, (-3.5, -2.0)),  # more blocks than warps: 4 to 16 chunks in front
])
def test_front_split_rules(n, W, H, log_scales):
    """A list's chunks composited by either pass: images within the rounding of a sum of n_contrib terms grouped by
    chunks of 32, against whole-list walks.  A pixel whose stop falls on the other side of the rounding differs by at most
    what the one that stopped left over."""
    import paper_2509_12138_gb300 as gs
    g = synth.random_gaussians(n, 0, 3, extent=1.0, log_scale_range=log_scales)
    cams = gs.pack_cameras(synth.orbital_cameras(8, 3.0, width=W, height=H).subset([0]))
    params = gs.pack_params(g, 0)
    fr = Frame(n, Units.single(n, 1), W, H, 0, with_backward=False, with_loss=False, chunk=32)
    fr.fit_capacity(params, cams)
    out = []
    for whole in (False, True):
        fr.walk_whole_lists = whole
        fr.preprocess(params, cams)
        fr.sort()
        fr.render((0.2, 0.4, 0.6))
        assert fr.read_status() == 0
        out.append((fr.img.double().cpu().reshape(3, -1), fr.final_T.double().cpu().reshape(-1),
                    fr.n_contrib.cpu().reshape(-1)))
    (ia, ta, na), (ib, tb, nb) = out
    same = na == nb
    colour = max(1.0, float(fr.rgb[:, :3].abs().max()))
    # T: a product of n_contrib factors, each pair of groupings n_contrib roundings apart; C: the sum of weights is 1
    eps = 2.0 ** -23 * (nb.double() + 64)
    assert float(same.double().mean()) > 0.99
    assert bool(((ta - tb).abs() <= eps * tb.clamp_min(1e-6))[same].all())
    assert bool(((ia - ib).abs() <= eps * colour)[:, same].all())
    assert bool(((ia - ib).abs() <= (2 * torch.maximum(ta, tb) + eps) * colour).all())


def _chunks_in_front(fr, K):
    """The M for which every list's 8x4-pixel blocks leave all chunks from M on to the parallel passes (no pixel stops;
    blocks past the image's edge have nothing to do)."""
    r = fr.ranges.cpu().numpy()
    nch = (r[:, 1] - r[:, 0] + K - 1) // K
    left = int(fr.stop_queue[-1])
    cols = np.clip((fr.W - 16 * np.arange(fr.TX) + 7) // 8, 0, 2)
    rows = np.clip((fr.H - 16 * np.arange(fr.TY) + 3) // 4, 0, 4)
    blocks = (rows[:, None] * cols).reshape(-1)
    fit = [m for m in range(1, 17) if int((blocks * np.maximum(nch - m, 0)).sum()) == left]
    assert fit, (left, nch.max())
    return nch, fit


@pytest.mark.parametrize("n,W,H,extent,log_scales,m", [
    (600, 64, 64, 3.0, (-3.5, -2.5), 16),      # lists of at most 8 chunks: all in front
    (4000, 32, 32, 3.0, (-3.5, -2.5), 1),      # covered, far fewer blocks than warps
    (12000, 64, 64, 3.0, (-3.5, -2.5), 1),
    (100000, 256, 256, 3.0, (-4.0, -3.0), 8),  # covered, about as many blocks as warps
    (30000, 200, 200, 0.5, (-3.8, -3.0), 1),   # fewer blocks than warps, empty lists
    (100000, 500, 500, 3.0, (-3.5, -2.5), None),  # more blocks than warps: 4 to 16
])
def test_front_split_by_lists(n, W, H, extent, log_scales, m):
    """How many chunks of 32 the front pass walks, read from the chunks it leaves to the passes behind it; splats so
    faint that no pixel stops."""
    import paper_2509_12138_gb300 as gs
    K = 32
    g = synth.random_gaussians(n, 0, 4, extent=extent, log_scale_range=log_scales)
    g["logit_opacity"][:] = -5.0
    cams = gs.pack_cameras(synth.orbital_cameras(8, 3.0, width=W, height=H).subset([0]))
    params = gs.pack_params(g, 0)
    fr = Frame(n, Units.single(n, 1), W, H, 0, with_backward=False, with_loss=False, chunk=K)
    fr.fit_capacity(params, cams)
    fr.forward(params, cams, (0.2, 0.4, 0.6))
    assert fr.read_status() == 0 and float(fr.final_T.min()) > 1e-3
    nch, fit = _chunks_in_front(fr, K)
    assert (nch.min() > 0) == (extent > 1.0)
    assert (nch.max() > 8) == (m != 16)
    assert m in fit if m else all(4 <= x <= 16 for x in fit)


@pytest.mark.parametrize("n,views,W,H,cap,lam,masks,whole", [
    (500, 1, 64, 64, None, 0.2, True, False), (300, 2, 64, 48, 1 << 15, 0.0, False, False),
    (20000, 1, 333, 250, None, 0.2, True, False), (20000, 1, 333, 250, None, 0.2, True, True),
    (4000, 1, 160, 160, 8000, 0.0, True, False), (300, 2, 1920, 1080, 1 << 15, 0.2, True, False),
    (300, 9, 1920, 1080, 1 << 15, 0.2, False, False)])
def test_launch_count_of_a_step(n, views, W, H, cap, lam, masks, whole):
    """The launches the benchmark reports for a step are those of a captured one, whatever its sizes make of it."""
    import paper_2509_12138_gb300 as gs
    g = synth.random_gaussians(n, 1, 8, extent=0.8, log_scale_range=(-4.0, -3.0))
    cams = gs.pack_cameras(synth.orbital_cameras(9, 3.0, width=W, height=H).subset(list(range(views))))
    params = gs.pack_params(g, 1)
    fr = Frame(n, Units.single(n, views), W, H, 1, max_instances=cap)
    if cap is None:
        fr.fit_capacity(params, cams)
    fr.use_masks, fr.walk_whole_lists = masks, whole
    gt, mask = torch.rand_like(fr.img), torch.ones((views, H, W), dtype=torch.uint8, device="cuda")
    opt = gs.Adam(params, 1)

    def step():
        fr.preprocess(params, cams)
        fr.sort()
        fr.render((1.0, 1.0, 1.0))
        fr.loss(gt, mask, lam)
        fr.blend_backward((1.0, 1.0, 1.0))
        opt.fused_step(fr, cams)

    assert captured_kernels(step) == bench.step_launch_count(fr, lam)
