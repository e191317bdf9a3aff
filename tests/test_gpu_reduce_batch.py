"""The sums of zm_errors and zm_errors_polar in launches of many images: as exact
as for one image, and the same bits whatever images share the launch.

Bar on a flat image, where the roundings of a lane's FP32 partial do not average
out: a lane adds at most a row's or run's trees of 256 pixels and nodes, so 16
steps for 3840 columns and 8 for 2048 nodes, after 4 roundings inside a tree,
and the warp's shuffle tree 5 more; the largest possible relative error of such
a sum is (16 + 4 + 5) 2^-24 = 1.5e-6.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2304_14492_gb300 import native as zm  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
BAR = 25 * 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2304_14492_gb300.build import build
    build()
    zm.lib()


def flat_ratio(f, g):
    """Eq. 10 of constant images f, g, and Eq. 13, in 64 bits."""
    d = float(np.float32(f) - np.float32(g))
    return d * d / (float(f) * float(f))


@pytest.mark.parametrize("h,w,batch", [(2160, 3840, 64), (2160, 3840, 128), (1080, 1920, 100), (64, 70, 128), (5000, 300, 9)])
def test_flat_images_in_one_launch(h, w, batch):
    f, g = np.float32(0.7361), np.float32(0.6113)
    ref = torch.full((h, w), float(f), device=DEV)
    tst = torch.full((h, w), float(g), device=DEV)
    err = torch.zeros((batch, 4), device=DEV, dtype=torch.float64)
    one = torch.zeros((1, 4), device=DEV, dtype=torch.float64)
    plan = zm.zm_plan(4, 8, 16)
    try:
        zm.zm_errors(plan, [ref] * batch, [tst] * batch, err)
        zm.zm_errors(plan, [ref], [tst], one)
        torch.cuda.synchronize()
    finally:
        zm.zm_plan_destroy(plan)
    assert torch.equal(err, one.expand(batch, 4))
    want = flat_ratio(f, g)
    e = one[0].cpu().numpy()
    assert abs(e[0] / want - 1.0) <= 2 * BAR and abs(e[1] / want - 1.0) <= BAR


@pytest.mark.parametrize("n_rho,n_theta,batch", [(1024, 1024, 32), (64, 64, 128), (37, 256, 130)])
def test_flat_nodes_in_one_launch(n_rho, n_theta, batch):
    f, g = np.float32(0.7361), np.float32(0.6113)
    a = torch.full((batch, n_rho, n_theta), float(f), device=DEV)
    b = torch.full((batch, n_rho, n_theta), float(g), device=DEV)
    err = torch.zeros((batch, 4), device=DEV, dtype=torch.float64)
    one = torch.zeros((1, 4), device=DEV, dtype=torch.float64)
    plan = zm.zm_plan(3, n_rho, n_theta)
    try:
        zm.zm_errors_polar(plan, a, b, batch, err)
        zm.zm_errors_polar(plan, a, b, 1, one)
        torch.cuda.synchronize()
    finally:
        zm.zm_plan_destroy(plan)
    assert torch.equal(err, one.expand(batch, 4))
    want = flat_ratio(f, g)
    e = one[0].cpu().numpy()
    assert e[3] == n_rho * n_theta and abs(e[0] / want - 1.0) <= 2 * BAR and abs(e[1] / want - 1.0) <= BAR


def test_images_of_many_heights_share_a_launch():
    rng = np.random.default_rng(3)
    sizes = [(1, 1), (7, 9), (8, 8), (9, 40), (65, 64), (400, 300), (2100, 31), (4200, 50)] * 17
    ims = {s: (torch.from_numpy(rng.random(s, dtype=np.float32) + 0.25).to(DEV),
               torch.from_numpy(rng.random(s, dtype=np.float32)).to(DEV)) for s in set(sizes)}
    err = torch.zeros((len(sizes), 4), device=DEV, dtype=torch.float64)
    one = torch.zeros((1, 4), device=DEV, dtype=torch.float64)
    mm = torch.zeros((len(sizes), 2), device=DEV)
    plan = zm.zm_plan(4, 8, 16)
    try:
        for _ in range(2):                                   # the second call finds the counters reset
            zm.zm_errors(plan, [ims[s][0] for s in sizes], [ims[s][1] for s in sizes], err)
            zm.zm_disk_minmax(plan, [ims[s][1] for s in sizes], mm)
        for s in ims:
            zm.zm_errors(plan, [ims[s][0]], [ims[s][1]], one)
            torch.cuda.synchronize()
            for b in (j for j, t in enumerate(sizes) if t == s):
                assert torch.equal(err[b], one[0]), s
                assert tuple(mm[b].tolist()) == tuple(mm[sizes.index(s)].tolist())
    finally:
        zm.zm_plan_destroy(plan)
