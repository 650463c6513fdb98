"""The one-ray-per-warp marches (small frames, ray batches, the batch of a
camera's rays that the device hands to the one-ray-per-thread form) against the
view marcher with one ray per thread (schedule "thread"): the same occupied
samples and early termination, and the same values up to the FP32 rounding of
two kernels that inline the same code (2e-6, as between the batched and the view
kernels)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2312_16457_gb300 import cow, synth
from gradcheck import assert_grad

pytestmark = pytest.mark.gpu
SAME = 2e-6


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2312_16457_gb300 import build

    build.build()
    oracle.build()
    torch.cuda.set_device(0)


def _scene(unbounded):
    if unbounded:
        sc, cams, mlp = synth.workload_unbounded(R=21, P=67, width=37, height=29)
        return sc, cams[0], mlp
    sc = synth.city_scene(23, 2, 2.0, [(21, 67)], **synth.SPARSE_CITY)
    return sc, synth.camera((-2.6, -3.1, 2.0), (0.3, 0.2, -0.8), 37, 29, 60.0), synth.mlp_weights(9)


def _same(got, want):
    assert torch.equal(got[2], want[2])
    assert float((got[0] - want[0]).abs().max()) <= SAME
    assert float((got[1] - want[1]).abs().max()) <= SAME


@pytest.mark.parametrize("ert", [0.0, 1e-2])
@pytest.mark.parametrize("form", ["fp32", "bf16_fp8", "fp8_bf16d bricks", "fp16 unbounded", "bf16 block_mlps"])
def test_warp_forms_equal_thread_form(form, ert):
    storage, *opt = form.split()
    sc, cam, mlp = _scene("unbounded" in opt)
    mlp = torch.from_numpy(mlp).cuda()
    ctx = cow.Context(sc, storage, bricks="bricks" in opt)
    bm = "block_mlps" in opt
    if bm:
        ctx.set_block_mlps(synth.block_mlp_weights(3, len(sc.blocks), 3), 3)
    ids = ctx.sort_blocks(cam, list(range(4)))
    kw = dict(ert_eps=ert, nsamp=True, block_mlps=bm)
    ctx.set_schedule("thread")
    want = ctx.render([cam], [ids], mlp, **kw)
    ctx.set_schedule("thread_const")
    _same(ctx.render([cam], [ids], mlp, **kw), want)
    o, d = (torch.from_numpy(x).cuda() for x in oracle.pixel_rays(cam))
    for n in (1, 3, 33, o.shape[0]):  # part of a CTA, a ray more than a warp of rays, all
        _same(ctx.render_rays(o[:n], d[:n], list(range(4)), mlp, **kw), [x[:n] for x in want])
    ctx.sync_check()
    assert int(want[2].max()) > 64  # several chunks of 32 samples
    ctx.close()


@pytest.mark.parametrize("order", ["coherent", "given"])
def test_camera_rays_equal_shuffled_rays(order):
    """2^17 rays and more: a camera's rays go to the thread form, the same rays
    shuffled to the warp form."""
    sc, cam, mlp = _scene(False)
    cam = synth.Camera(cam.c2w, 512, 300, cam.fov_y_deg)
    ctx = cow.Context(sc, "bf16")
    ctx.set_ray_order(order)
    ctx.set_schedule("thread")
    ids = ctx.sort_blocks(cam, list(range(4)))
    mlp = torch.from_numpy(mlp).cuda()
    want = ctx.render([cam], [ids], mlp, ert_eps=1e-3, nsamp=True)
    o, d = (torch.from_numpy(x).cuda() for x in oracle.pixel_rays(cam))
    _same(ctx.render_rays(o, d, list(range(4)), mlp, ert_eps=1e-3, nsamp=True), want)
    perm = torch.randperm(o.shape[0], generator=torch.Generator().manual_seed(1)).cuda()
    got = ctx.render_rays(o[perm], d[perm], list(range(4)), mlp, ert_eps=1e-3, nsamp=True)
    _same(got, [x[perm] for x in want])
    ctx.sync_check()
    ctx.close()


@pytest.mark.parametrize("n_ids", [33, 64])
def test_block_order_beyond_a_warp(n_ids):
    """More blocks than lanes: per-ray order, culling and per-block outputs
    against the oracle."""
    sc = synth.city_scene(29, 8, 2.0, [(6, 10)])
    o, d = synth.random_rays(257, 5, sc.box_lo, sc.box_hi)
    mlp = synth.mlp_weights(2)
    ctx = cow.Context(sc, "fp32")
    ids = list(np.random.default_rng(1).permutation(64)[:n_ids])
    rgb, aux, ns = ctx.render_rays(o.cuda(), d.cuda(), ids, mlp, nsamp=True)
    _, aux_t, bt = ctx.render_rays_block_t(o.cuda(), d.cuda(), ids, mlp)
    part = ctx.render_partials(o.cuda(), d.cuda(), ids)
    ctx.sync_check()
    r_o, a_o, n_o = oracle.render_rays(oracle.OracleScene(sc), ids, o, d, mlp)
    assert np.array_equal(ns.cpu().numpy(), n_o)
    assert np.abs(rgb.cpu().numpy() - r_o).max() <= 1e-4
    assert np.abs(aux.cpu().numpy() - a_o).max() <= 1e-4
    assert torch.equal(aux_t, aux)
    hit = bt >= 0
    assert torch.equal(hit.any(1), ns > 0) and float((part[..., 7] - torch.where(hit, bt, 1.0)).abs().max()) <= SAME
    assert float((torch.where(hit, bt, 1.0).prod(1) - aux[:, 7]).abs().max()) <= 1e-5
    ctx.close()


@pytest.mark.parametrize("form", ["fp32", "bf16", "fp16 unbounded"])
def test_backward_edges(form):
    """The cooperative scatter at partial chunks and CTAs, odd resolutions and
    contracted blocks: 300 rays at once against the oracle's gradient, and the
    same rays in calls of 1, 5, 33 and 261 against that up to the order of the
    FP32 reductions (1e-5 of each array's largest entry); arrays that are not
    asked for stay out of it."""
    storage, *opt = form.split()
    n = 300
    sc, _, mlp = _scene("unbounded" in opt)
    o, d = synth.random_rays(n, 12, sc.box_lo, sc.box_hi)
    if "unbounded" in opt:
        o = torch.tensor([0.25, -0.4, 0.3]).expand(n, 3).contiguous()
    g = np.random.default_rng(6).normal(size=(n, 3)).astype(np.float32)
    ctx = cow.Context(sc, storage)
    ids = list(range(4))
    oc, dc, gc, mc = o.cuda(), d.cuda(), torch.from_numpy(g).cuda(), torch.from_numpy(mlp).cuda()
    _, aux, _ = ctx.render_rays(oc, dc, ids, mc)
    res = []
    for cuts in ((0, n), (0, 1, 6, 39, n)):
        gg = [torch.zeros(b.grid.shape, device="cuda") for b in sc.blocks]
        gp = [[torch.zeros(p.shape, device="cuda") for p in b.planes] for b in sc.blocks]
        gm = torch.zeros(499, device="cuda")
        ga, pa = list(gg), [list(p) for p in gp]
        if len(cuts) > 2:  # without block 1's grid and block 2's xz plane
            ga[1], pa[2][1] = None, None
        for a, b in zip(cuts, cuts[1:]):
            ctx.render_backward(oc[a:b], dc[a:b], ids, mc, aux[a:b], gc[a:b], ga, pa, gm)
        ctx.sync_check()
        res.append((gg, gp, gm))
    og, op, om = oracle.render_rays_grad(
        oracle.OracleScene(sc, values="master" if storage == "fp32" else storage), ids, o, d, mlp, g)
    (gg, gp, gm), (sg, sp, sm) = res
    assert_grad(gm, om, "mlp")

    def close(x, y):
        assert float((x - y).abs().max()) <= 1e-5 * float(y.abs().max())

    close(sm, gm)
    for b in range(4):
        assert_grad(gg[b], og[b], f"grid {b}")
        close(sg[b], gg[b] * (b != 1))
        for k in range(3):
            assert_grad(gp[b][k], op[b][k], f"plane {b} {k}")
            close(sp[b][k], gp[b][k] * ((b, k) != (2, 1)))
    ctx.close()
