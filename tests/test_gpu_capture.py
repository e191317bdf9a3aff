"""Calls captured into a CUDA graph after a warm-up that took another path: a call
of few samples gathers and builds nothing, one of many resamples by tiles or from
staged rows and needs the geometry's work list."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2304_14492_gb300 import native as zm  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2304_14492_gb300.build import build
    build()
    zm.lib()


# warm-up batch, captured batch: 256 angles, gathered / staged (also from above the
# staged window); 512 and 1024 angles, gathered / tiles; nothing warmed up
@pytest.mark.parametrize("prec", [zm.ZM_PREC_FP32, zm.ZM_PREC_BF16X3])
@pytest.mark.parametrize("side,n_max,n_rho,n_theta,warm,batch",
                         [(512, 50, 256, 256, 1, 16), (512, 50, 256, 256, 40, 16), (512, 100, 256, 512, 1, 16),
                          (1024, 100, 512, 1024, 1, 8), (512, 100, 256, 512, 0, 16)])
def test_captured_batch_differs_from_the_warm_up(side, n_max, n_rho, n_theta, warm, batch, prec):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(side + n_theta)
    most = max(warm, batch)
    imgs = [torch.rand((side, side), device=DEV, generator=gen) for _ in range(most)]
    arr = zm.image_array(imgs[:batch])
    P = zm.zm_num_moments(n_max)
    out = torch.full((most, P, 2), float("nan"), device=DEV)
    plan = zm.zm_plan(n_max, n_rho, n_theta, prec)
    try:
        zm.zm_plan_reserve(plan, most)
        side_stream = torch.cuda.Stream()
        with torch.cuda.stream(side_stream):
            if warm:
                zm.zm_moments(plan, imgs[:warm], out)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side_stream):
            zm.zm_moments(plan, arr, out)
        out.fill_(float("nan"))
        for im in imgs:
            im.mul_(0.5)                                     # the graph reads the images of its replay
        graph.replay()
        torch.cuda.synchronize()
        got = out[:batch].clone()
        zm.zm_moments(plan, arr, out)
        zm.zm_plan_status(plan)
        assert torch.isfinite(got).all() and torch.equal(got, out[:batch])
    finally:
        zm.zm_plan_destroy(plan)
