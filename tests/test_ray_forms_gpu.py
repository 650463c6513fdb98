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
