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
