"""Deterministic mode: the screen-space gradients accumulate as int64 fixed point, whose sums do not depend on
the order in which warps add them, so a training step is bitwise reproducible run to run and across a
checkpoint / resume, and it agrees with the float-atomic path and with the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2509_12138_gb300 as gs
from tests import scenes
from tests.gpu_util import gauss64
from paper_2509_12138_gb300 import workload
from paper_2509_12138_gb300.train import BatchedTrainer, PlainTrainer, split_views

pytestmark = pytest.mark.gpu
BG = (1.0, 1.0, 1.0)


def _grads(g, cams, deg, W, H, deterministic, chunk=1024):
    n = g["means"].shape[0]
    params = gs.pack_params(g, deg)
    camd = gs.pack_cameras(cams)
    gt, mask = scenes.random_gt(W, H, 9)
    fr = gs.Frame(n, gs.Units.single(n), W, H, deg, deterministic=deterministic, chunk=chunk)
    fr.fit_capacity(params, camd)
    fr.forward(params, camd, BG)
    fr.loss(torch.from_numpy(gt).cuda()[None], torch.from_numpy(mask).cuda()[None], 0.2)
    grads = fr.backward(params, camd, BG)
    torch.cuda.synchronize()
    assert fr.read_status() == 0
    return grads.clone(), torch.cat([fr.dxy, fr.dco, fr.drgb], 1).clone()


@pytest.mark.parametrize("chunk", [1024, 32])
def test_gradients_bitwise_reproducible(chunk):
    # dense, overlapping splats: many warps add to the same records in an order that varies run to run
    g, cams = scenes.random_scene(4000, 2, 81, 160, 120, log_scale_range=(-3.0, -2.0))
    a = _grads(g, cams, 2, 160, 120, True, chunk)
    b = _grads(g, cams, 2, 160, 120, True, chunk)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert float(a[0].abs().max()) > 0


def test_deterministic_agrees_with_float_path_and_oracle():
    deg, W, H = 1, 96, 80
    g, cams = scenes.random_scene(1200, deg, 82, W, H)
    d, d2 = _grads(g, cams, deg, W, H, True)
    f, f2 = _grads(g, cams, deg, W, H, False)
    sc = float(f.abs().max())
    assert torch.allclose(d, f, rtol=1e-4, atol=1e-5 * sc)
    assert torch.allclose(d2, f2, rtol=1e-4, atol=1e-5 * float(f2.abs().max()))
    # against the oracle's gradient of the same loss
    gt, mask = scenes.random_gt(W, H, 9)
    cam = oracle.camera_block(cams, 0)
    r = oracle.render(gauss64(g), cam, BG)
    _, dimg = oracle.loss(r["img"], gt.astype(np.float64), mask, 0.2)
    go = oracle.project_backward(gauss64(g), cam, oracle.render_backward(gauss64(g), cam, BG, dimg))
    gg = gs.unpack_grads(d, deg)
    for sl in (slice(0, 3), slice(3, 6), slice(6, 10), slice(10, 11), slice(11, 14)):
        ref = go[:, sl]
        assert np.abs(gg[:, sl] - ref).max() <= 1e-3 * np.abs(ref).max()


def _small_scene():
    return workload.isosurface_scene(30000, 4, 8, 128, 96, sh_degree=1, seed=5)


@pytest.mark.parametrize("on_disk", [False, True])
def test_checkpoint_resume_is_bitwise_identical(on_disk, tmp_path):
    """A run resumed from a checkpoint (in memory, or through the on-disk file format) continues bit for bit
    like the uninterrupted run."""
    scene = _small_scene()
    train_v, _ = split_views(len(scene.cams))

    def trainer():
        p = gs.pack_params(scene.init, scene.sh_degree)
        return PlainTrainer(p, scene.sh_degree, scene.cams_dev, scene.gt, scene.mask, train_v, deterministic=True,
                            seed=3)

    a = trainer()
    for _ in range(6):
        a.step()
    b = trainer()
    for _ in range(3):
        b.step()
    c = trainer()  # a fresh process would start here from the checkpoint
    if on_disk:
        path = str(tmp_path / "resume.ckpt")
        b.save(path)
        del b
        c.load(path)
    else:
        c.load_state_dict(b.state_dict())
    for _ in range(3):
        c.step()
    torch.cuda.synchronize()
    assert a.check() == 0 and c.check() == 0
    assert torch.equal(a.params, c.params)
    assert torch.equal(a.opt.m, c.opt.m) and torch.equal(a.opt.v, c.opt.v)
    assert int(a.opt.step_dev.item()) == int(c.opt.step_dev.item()) == 6
    assert not torch.equal(a.params, gs.pack_params(scene.init, scene.sh_degree))  # training moved them


def test_graph_captured_batched_training_is_bitwise_reproducible():
    ps = workload.partitioned_scene([8000, 16000, 12000], 4, 8, 96, 72, n_parts=3, ghost=0.05, sh_degree=1)
    train_v, _ = split_views(8)
    runs = []
    for _ in range(2):
        p = gs.pack_params(ps.init, 1)
        tr = BatchedTrainer(p, 1, ps.offsets, ps.cams_dev, ps.gt, ps.mask, train_v, views_per_step=2,
                            deterministic=True)
        for _ in range(5):
            tr.step()
        torch.cuda.synchronize()
        assert tr.check() == 0
        runs.append((p.clone(), tr.opt.m.clone()))
    assert torch.equal(runs[0][0], runs[1][0]) and torch.equal(runs[0][1], runs[1][1])


@pytest.mark.parametrize("n", [1, 2, 8, 9, 33, 70])
@pytest.mark.parametrize("variant", [0, 1, 2])
def test_deterministic_gradients_of_few_hits(n, variant):
    """Lists of a few entries and just over: both ways of summing a hit over a block's pixels agree with the float
    path (bounds as above), for every block shape, ragged image edges and a pixel that stops inside a batch."""
    W, H = 43, 38
    g, cams = scenes.random_scene(n, 1, 90 + n, W, H, log_scale_range=(-2.5, -1.0))
    g["logit_opacity"][:] = np.where(np.arange(n) % 3 == 0, 6.0, 0.0)
    params, camd = gs.pack_params(g, 1), gs.pack_cameras(cams)
    gt, mask = scenes.random_gt(W, H, 9)
    out = []
    for deterministic in (True, True, False):
        fr = gs.Frame(n, gs.Units.single(n), W, H, 1, deterministic=deterministic, variant=variant, chunk=32)
        fr.fit_capacity(params, camd)
        fr.forward(params, camd, BG)
        fr.loss(torch.from_numpy(gt).cuda()[None], torch.from_numpy(mask).cuda()[None], 0.2)
        fr.backward(params, camd, BG)
        torch.cuda.synchronize()
        assert fr.read_status() == 0
        out.append([fr.dxy.clone(), fr.dco.clone(), fr.drgb.clone()])
    assert all(torch.equal(a, b) for a, b in zip(out[0], out[1]))
    assert all(float(f.abs().max()) > 0 for f in out[2])
    for d, f in zip(out[0], out[2]):
        assert torch.allclose(d, f, rtol=1e-4, atol=1e-5 * float(f.abs().max()))
