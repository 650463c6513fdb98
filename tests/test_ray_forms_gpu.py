"""Ray batches and views in their two forms, one ray per warp and one ray per
thread: which form a call takes, and that the form does not show in the
results."""
import numpy as np
import pytest
import torch

import oracle
from paper_2312_16457_gb300 import cow, synth

pytestmark = pytest.mark.gpu
IDS = list(range(4))


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2312_16457_gb300 import build

    build.build()
    oracle.build()
    torch.cuda.set_device(0)


def _city():
    return synth.city_scene(23, 2, 2.0, [(21, 67)], **synth.SPARSE_CITY)


def _camera_rays(w, h):
    cam = synth.camera((-2.6, -3.1, 2.0), (0.3, 0.2, -0.8), w, h, 60.0)
    return [torch.from_numpy(x).cuda() for x in oracle.pixel_rays(cam)]


def test_given_order_needs_no_scratch_and_its_graph_stands_alone():
    """A batch in the given order allocates nothing, and a graph of one still
    renders after a larger batch."""
    sc, mlp = _city(), torch.from_numpy(synth.mlp_weights(9)).cuda()
    o, d = _camera_rays(512, 300)
    big = [x.repeat(5, 1) for x in (o, d)]
    first = cow.Context(sc, "bf16")  # loads the kernels and fills torch's pool
    for order in ("coherent", "given"):
        first.set_ray_order(order)
        want = first.render_rays(o, d, IDS, mlp, ert_eps=1e-3)
        first.render_rays(*big, IDS, mlp, ert_eps=1e-3)
    first.sync_check()
    ctx = cow.Context(sc, "bf16")
    ctx.set_ray_order("given")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx.render_rays(o, d, IDS, mlp, ert_eps=1e-3)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        got = ctx.render_rays(o, d, IDS, mlp, ert_eps=1e-3)
    ctx.set_ray_order("coherent")
    ctx.render_rays(*big, IDS, mlp, ert_eps=1e-3)
    for _ in range(2):
        got[0].zero_()
        g.replay()
        ctx.sync_check()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    ctx.close()
    first.close()


@pytest.mark.parametrize("block_mlps", [False, True])
def test_early_termination_in_front_of_nan_features(block_mlps):
    """Features that are NaN behind an opaque layer, fewer samples behind it
    than a warp takes at once: a ray that ends in the layer never reads them,
    in the colours, the sample counts and the gradients."""
    R, P, n = 17, 64, 65
    clean = torch.full((R, R, R, 8), 0.25)
    clean[..., 0] = -10.0
    clean[8, ..., 0] = 8.0  # [z, y, x]: the layer
    nan = clean.clone()
    nan[4:6] = float("nan")
    planes = [torch.zeros(P, P, 8) for _ in range(3)]
    sc = synth.Scene([synth.Block((-1.0,) * 3, (1.0,) * 3, R, P, 1, -1, clean, planes)], (-1.0,) * 3, (1.0,) * 3, [0.0])
    gen = torch.Generator().manual_seed(4)
    o = torch.cat([torch.rand((n, 2), generator=gen) - 0.5, torch.full((n, 1), 2.0)], 1).cuda()
    d = torch.nn.functional.normalize(torch.cat([0.1 * torch.rand((n, 2), generator=gen), -torch.ones(n, 1)], 1)).cuda()
    mlp = torch.from_numpy(synth.mlp_weights(2)).cuda()
    g = torch.rand((n, 3), generator=gen).cuda()
    cam, out = synth.camera((0.0, -0.1, 2.5), (0.0, 0.0, 0.0), 9, 7, 20.0), []
    ctx = cow.Context(sc, "fp32")
    if block_mlps:
        ctx.set_block_mlps(synth.block_mlp_weights(3, 1, 2), 2)
    for grid in (clean, nan):
        ctx.update_features(0, grid.cuda(), [p.cuda() for p in planes])
        kw = dict(ert_eps=1e-3, nsamp=True, block_mlps=block_mlps)
        res = [*ctx.render([cam], [[0]], mlp, **kw), *ctx.render_rays(o, d, [0], mlp, **kw)]
        if not block_mlps:
            gg, gp = torch.zeros(R, R, R, 8).cuda(), [torch.zeros(P, P, 8).cuda() for _ in range(3)]
            ctx.render_backward(o, d, [0], mlp, res[4], g, [gg], [gp], torch.zeros(499).cuda(), ert_eps=1e-3)
            assert float(gg.abs().max()) > 0
            res += [gg, *gp]
        ctx.sync_check()
        out.append(res)
    for k, (a, b) in enumerate(zip(*out)):
        if k < 6:
            assert torch.equal(a, b)
        else:  # sums of up to 65 rays in any order
            assert float((a - b).abs().max()) <= 1e-5 * float(a.abs().max())
    assert int(out[0][5].min()) > 8
    ctx.close()


FORMS = ["fp32", "fp16", "bf16_fp8", "fp8 bricks", "fp8_bf16d bricks", "fp16 unbounded"]


def _scene(opt):
    if "unbounded" in opt:
        return synth.workload_unbounded(R=21, P=67, width=37, height=29)[0]
    return _city()


def _rays(opt, sc, n):
    o, d = synth.random_rays(n, 12, sc.box_lo, sc.box_hi)
    if "unbounded" in opt:
        o = torch.tensor([0.25, -0.4, 0.3]).expand(n, 3).contiguous()
    return o.cuda(), d.cuda()


def _marches(ctx, sc, o, d, mlp, ids):
    """Every ray call that chooses a form: (the form, outputs, in-block
    transmittances, opacity gradients)."""
    out = list(ctx.render_rays(o, d, ids, mlp, ert_eps=1e-2, nsamp=True))
    out += list(ctx.render_rays(o, d, ids, None, ert_eps=1e-2, nsamp=True, block_mlps=True))
    out += [*ctx.render_rays_block_t(o, d, ids, mlp)[:2], *ctx.render_rays_block_state(o, d, ids)]
    out.append(ctx.render_partials(o, d, ids))
    form = ctx.last_form()
    bt = ctx.render_rays_block_t(o, d, ids, mlp)[2]
    grads = []
    for T in (None, bt):
        gg = [torch.zeros(b.grid.shape, device="cuda") for b in sc.blocks]
        gp = [[torch.zeros(p.shape, device="cuda") for p in b.planes] for b in sc.blocks]
        grads.append([ctx.opacity_loss(o, d, ids, 0.5, grads=(gg, gp), block_T=T), *gg, *sum(gp, [])])
    return form, out, bt, grads


@pytest.mark.parametrize("form", FORMS)
def test_ray_calls_do_not_depend_on_the_form(form):
    """Every march of a ray batch in both forms: outputs, sample counts and
    per-block states bit for bit; what is summed in another order (the optical
    depth of a block, the opacity loss and its gradient) to FP32 rounding."""
    storage, *opt = form.split()
    sc = _scene(opt)
    o, d = _rays(opt, sc, 1003)
    mlp = torch.from_numpy(synth.mlp_weights(9)).cuda()
    ctx = cow.Context(sc, storage, bricks="bricks" in opt)
    ctx.set_block_mlps(synth.block_mlp_weights(3, 4, 2), 2)
    res = []
    for f in ("thread", "warp"):
        ctx.set_test_hooks(form=f)
        res.append(_marches(ctx, sc, o, d, mlp, IDS))
        assert res[-1][0] == f
    ctx.set_test_hooks()
    ctx.sync_check()
    (_, a, bt_a, ga), (_, b, bt_b, gb) = res
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    assert torch.equal(bt_a < 0, bt_b < 0) and int((bt_a >= 0).sum()) > 500
    # exp(-tau): tau of up to ~300 samples, whose 32 lane sums carry some 10 roundings
    # of a partial sum each: 2^-24 (10 + 5) tau exp(-tau) at most, tau exp(-tau) <= 0.37
    assert float((bt_a - bt_b).abs().max()) <= 5e-7
    for x, y in zip(ga, gb):
        for u, v in zip(x, y):
            assert float((u - v).abs().max()) <= 1e-4 * float(v.abs().max()) + 1e-12
    ctx.close()


@pytest.mark.parametrize("order", ["coherent", "given"])
@pytest.mark.parametrize("form", ["fp32", "bf16_fp8", "fp8 bricks"])
def test_camera_rays_take_the_thread_form(form, order):
    """A camera's 2^17 rays and more (not a whole number of CTAs) take the thread
    form in every march, the same rays shuffled the warp form, with the same
    results, also where only seven tenths of the rays are the camera's."""
    storage, *opt = form.split()
    sc = synth.city_scene(23, 2, 2.0, [(21, 260)], **synth.SPARSE_CITY)
    mlp = torch.from_numpy(synth.mlp_weights(9)).cuda()
    ctx = cow.Context(sc, storage, bricks="bricks" in opt)
    ctx.set_block_mlps(synth.block_mlp_weights(3, 4, 2), 2)
    ctx.set_ray_order(order)
    o, d = _camera_rays(500, 301)
    n = o.shape[0]
    perm = torch.randperm(n, generator=torch.Generator().manual_seed(1)).cuda()
    mixed = torch.cat([torch.arange(n * 7 // 10, device="cuda"), perm[perm >= n * 7 // 10]])
    calls = [lambda o, d: ctx.render_rays(o, d, IDS, mlp, ert_eps=1e-3, nsamp=True),
             lambda o, d: ctx.render_rays(o, d, IDS, None, ert_eps=1e-3, nsamp=True, block_mlps=True),
             lambda o, d: ctx.render_rays_block_t(o, d, IDS, mlp)[:2],
             lambda o, d: ctx.render_rays_block_state(o, d, IDS),
             lambda o, d: [ctx.render_partials(o, d, IDS)]]
    for call in calls:
        want = call(o, d)
        assert ctx.last_form() == "thread"
        for p in (perm, mixed):
            got = call(o[p], d[p])
            assert ctx.last_form() == "warp"
            for x, y in zip(got, want):
                assert torch.equal(x, y[p])
    loss = ctx.opacity_loss(o, d, IDS)
    gg = [torch.zeros(b.grid.shape, device="cuda") for b in sc.blocks]
    gp = [[torch.zeros(p.shape, device="cuda") for p in b.planes] for b in sc.blocks]
    ctx.render_backward(o[perm], d[perm], IDS, mlp, torch.zeros(n, 8, device="cuda"), torch.zeros(n, 3, device="cuda"),
                        gg, gp, torch.zeros(499, device="cuda"))
    assert ctx.last_form() == "thread"  # the opacity call's, whatever was ordered since
    again = ctx.opacity_loss(o[perm], d[perm], IDS)
    assert ctx.last_form() == "warp"
    assert abs(float(loss) - float(again)) <= 1e-5 * float(loss)
    ctx.sync_check()
    ctx.close()


@pytest.mark.parametrize("form", ["fp32", "fp16 unbounded"])
def test_gradients_of_camera_rays_with_the_thread_forms_totals(form):
    """The backward of a camera's rays takes its totals from the thread form and
    marches one ray per warp: the same gradients as with the warp form's totals,
    and as the sum in 64 bits over 64 calls."""
    storage, *opt = form.split()
    sc = _scene(opt)
    mlp = torch.from_numpy(synth.mlp_weights(9)).cuda()
    ctx = cow.Context(sc, storage)
    o, d = _camera_rays(500, 301)
    if "unbounded" in opt:
        o = o + torch.tensor([2.6, 3.1, -1.6], device="cuda")
    n = o.shape[0]
    g = torch.randn((n, 3), generator=torch.Generator().manual_seed(2)).cuda() / n

    def grad(part, aux):
        gg = [torch.zeros(b.grid.shape, device="cuda") for b in sc.blocks]
        gp = [[torch.zeros(p.shape, device="cuda") for p in b.planes] for b in sc.blocks]
        gm = torch.zeros(499, device="cuda")
        ctx.render_backward(o[part], d[part], IDS, mlp, aux[part], g[part], gg, gp, gm)
        return [gm, *gg, *sum(gp, [])]

    auxs = []
    for f in ("thread", "warp"):
        ctx.set_test_hooks(form=f)
        auxs.append(ctx.render_rays(o, d, IDS, mlp)[1])
    ctx.set_test_hooks()
    assert torch.equal(*auxs)
    got, want = grad(slice(None), auxs[0]), None
    for k in range(64):
        part = [x.double() for x in grad(slice(k * n // 64, (k + 1) * n // 64), auxs[0])]
        want = part if want is None else [a + b for a, b in zip(want, part)]
    ctx.sync_check()
    for a, b in zip(got, want):
        assert float((a.double() - b).abs().max()) <= 1e-4 * float(b.abs().max())
    ctx.close()


@pytest.mark.parametrize("ert", [0.0, 1e-2])
@pytest.mark.parametrize("form", FORMS + ["bf16 block_mlps"])
def test_views_do_not_depend_on_the_form(form, ert):
    storage, *opt = form.split()
    sc = _scene(opt)
    ctx = cow.Context(sc, storage, bricks="bricks" in opt)
    bm = "block_mlps" in opt
    if bm:
        ctx.set_block_mlps(synth.block_mlp_weights(3, 4, 3), 3)
    cam = synth.camera((-0.6, -0.5, 0.6) if "unbounded" in opt else (-2.6, -3.1, 2.0), (0.9, 0.8, -0.5), 37, 29, 60.0)
    ids = ctx.sort_blocks(cam, IDS)
    res = []
    for f in ("thread", "warp"):
        ctx.set_test_hooks(form=f)
        res.append(ctx.render([cam], [ids], synth.mlp_weights(9), ert_eps=ert, nsamp=True, block_mlps=bm))
        assert ctx.last_form() == f
    ctx.set_test_hooks()
    ctx.sync_check()
    for x, y in zip(*res):
        assert torch.equal(x, y)
    assert int(res[0][2].max()) > 64
    ctx.close()


def test_small_planes_take_the_thread_form_earlier():
    """Few samples a ray: frames and batches take the thread form where the same
    calls over larger planes take the warp form."""
    mlp = torch.from_numpy(synth.mlp_weights(9)).cuda()
    form = {}
    for P in (33, 260):
        sc = synth.single_block_scene(1, 9, P)
        ctx = cow.Context(sc, "bf16")
        cam = synth.camera((0.0, -2.5, 0.8), (0.0, 0.0, 0.0), 200, 150, 60.0)
        ctx.render([cam], [[0]], mlp)
        form["view", P] = ctx.last_form()
        o, d = (torch.from_numpy(x).cuda() for x in oracle.pixel_rays(cam))
        perm = torch.randperm(o.shape[0], generator=torch.Generator().manual_seed(1)).cuda()
        for name, p in (("camera", slice(None)), ("random", perm)):
            res = []
            for f in (None, "warp"):
                ctx.set_test_hooks(form=f)
                res.append(ctx.render_rays(o[p], d[p], [0], mlp, nsamp=True))
                if f is None:
                    form[name, P] = ctx.last_form()
            for x, y in zip(*res):
                assert torch.equal(x, y)
        ctx.sync_check()
        ctx.close()
    assert form == {(k, P): "thread" if P == 33 else "warp" for P in (33, 260) for k in ("view", "camera", "random")}


def test_unbounded_blocks_take_the_thread_form_earlier():
    """Contracted blocks: frames and batches from some 20000 rays on."""
    mlp = torch.from_numpy(synth.mlp_weights(9)).cuda()
    sc, cams, _ = synth.workload_unbounded(R=9, P=260)
    form = {}
    for flags in (True, False):
        ctx = cow.Context(sc, "bf16")
        if not flags:
            for i in IDS:
                ctx.set_unbounded(i, 0)
        for w, h in ((120, 100), (250, 200)):
            cam = synth.Camera(cams[0].c2w, w, h, 70.0)
            ctx.render([cam], [ctx.sort_blocks(cam, IDS)], mlp)
            form["view", flags, w] = ctx.last_form()
            o, d = (torch.from_numpy(x).cuda() for x in oracle.pixel_rays(cam))
            perm = torch.randperm(w * h, generator=torch.Generator().manual_seed(1)).cuda()
            o, d = o[perm], d[perm]
            for name, call in (("march", lambda: ctx.render_rays(o, d, IDS, mlp)),
                               ("partials", lambda: ctx.render_partials(o, d, IDS)),
                               ("opacity", lambda: ctx.opacity_loss(o, d, IDS))):
                call()
                form[name, flags, w] = ctx.last_form()
        ctx.sync_check()
        ctx.close()
    assert form == {(k, u, w): "thread" if u and w == 250 else "warp" for k in ("view", "march", "partials", "opacity")
                    for u in (True, False) for w in (120, 250)}


@pytest.mark.parametrize("order", ["coherent", "given"])
def test_opacity_gradient_with_a_thread_form_first_march(order):
    """A camera's rays: the transmittances of the first march come from the thread
    form, the scatter runs one ray per warp.  The same loss and gradient as from
    the forward's transmittances, summed in 64 bits over 64 calls."""
    sc = synth.city_scene(23, 2, 2.0, [(66, 260)], **synth.SPARSE_CITY)
    mlp = torch.from_numpy(synth.mlp_weights(9)).cuda()
    ctx = cow.Context(sc, "bf16")
    ctx.set_ray_order(order)
    o, d = _camera_rays(500, 301)
    n = o.shape[0]

    def term(part, T):
        gg = [torch.zeros(b.grid.shape, device="cuda") for b in sc.blocks]
        gp = [[torch.zeros(p.shape, device="cuda") for p in b.planes] for b in sc.blocks]
        k = o[part].shape[0]
        loss = ctx.opacity_loss(o[part], d[part], IDS, weight=k / n, grads=(gg, gp), block_T=T)
        return [loss, *gg, *sum(gp, [])]

    got = term(slice(None), None)
    assert ctx.last_form() == "thread"
    ctx.set_test_hooks(form="thread")
    T, want = ctx.render_rays_block_t(o, d, IDS, mlp)[2], None
    for k in range(64):
        part = slice(k * n // 64, (k + 1) * n // 64)
        x = [y.double() for y in term(part, T[part].contiguous())]
        assert ctx.last_form() == "warp"
        want = x if want is None else [a + b for a, b in zip(want, x)]
    ctx.sync_check()
    # T of both marches: expf against __expf of the log-density and its product, some
    # 1e-6 tau relative; where T nears the clamp at 1e-6 (tau = 14) the gradient's
    # log(1 - alpha) and its rounding take up to 1e-2 of a single ray's share, the
    # largest entry sums hundreds of rays
    for a, b in zip(got, want):
        assert float((a.double() - b).abs().max()) <= 1e-3 * float(b.abs().max())
    ctx.close()


@pytest.mark.parametrize("ert", [0.0, 1e-2])
@pytest.mark.parametrize("storage", ["fp32", "fp8_bf16d"])
def test_warp_schedule_of_odd_frames(storage, ert):
    """COW_SCHED_WARP: warps whose 32 pixels lie partly outside the frame."""
    ctx = cow.Context(_city(), storage)
    res = []
    cams = [synth.camera((-2.6, -3.1, 2.0), (0.3, 0.2, -0.8), w, h, 60.0) for w, h in ((37, 29), (1, 1), (16, 9))]
    ids = [ctx.sort_blocks(c, IDS) for c in cams]
    for sched, form in (("thread", "thread"), ("warp", "warp")):
        ctx.set_schedule(sched)
        res.append(ctx.render(cams, ids, synth.mlp_weights(9), ert_eps=ert, nsamp=True))
        assert ctx.last_form() == form
    ctx.sync_check()
    for x, y in zip(*res):
        assert torch.equal(x, y)
    ctx.close()
