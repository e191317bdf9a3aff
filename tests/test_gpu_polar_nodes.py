"""Polar to pixels on grids of many nodes, whose place in the table is guessed from a
closed form and confirmed: one canvas (its own kernel) and several of one size give
the same pixels, and both agree with the oracle's interpolation.

Bar: the radial fraction and theta N / 2 pi carry a few FP32 roundings of values up to
N and N_rho, hence 8 * 2^-24 * max(N, N_rho) of a sample step, at most 2 max |f| in
each direction; Gauss nodes near the rim are denser by the ratio of the largest spacing
to the smallest.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import grid, metrics, reconstruct as orc  # noqa: E402
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


@pytest.mark.parametrize("gauss", [False, True])
@pytest.mark.parametrize("n_rho,n_theta,h,w", [(1, 8, 20, 21), (3, 8, 33, 40), (64, 64, 301, 257), (777, 64, 200, 200),
                                               (2048, 16, 180, 150)])
def test_one_canvas_and_several(n_rho, n_theta, h, w, gauss):
    P = zm.zm_num_moments(3)
    rng = np.random.default_rng(n_rho)
    z = torch.from_numpy(rng.uniform(-0.05, 0.05, (1, P, 2)).astype(np.float32)).to(DEV)
    one = torch.full((h, w), 7.0, device=DEV)
    many = [torch.full((h, w), 7.0, device=DEV) for _ in range(3)]
    polar = torch.empty((3, n_rho, n_theta), device=DEV)
    plan = zm.zm_plan(3, n_rho, n_theta, zm.ZM_GRID_GAUSS if gauss else 0)
    try:
        zm.zm_reconstruct_cartesian(plan, z, [one], polar, zm.ZM_NEUMANN)
        zm.zm_reconstruct_cartesian(plan, z.expand(3, P, 2).contiguous(), many, polar, zm.ZM_NEUMANN)
        torch.cuda.synchronize()
    finally:
        zm.zm_plan_destroy(plan)
    assert all(torch.equal(c, one) for c in many)
    rho, _ = grid.radial_nodes(n_rho, "gauss" if gauss else "midpoint")
    ref = orc.polar_to_cartesian(polar[0].double().cpu().numpy(), rho, h, w)
    steps = np.diff(rho)
    dense = steps.max() / steps.min() if n_rho > 1 else 1.0
    bar = 4 * 8 * 2.0 ** -24 * max(n_rho * dense, n_theta, 8) * float(polar.abs().max())
    got = one.double().cpu().numpy()
    mask = metrics.disk_mask(h, w)
    assert np.all(got[~mask] == 0.0) and np.max(np.abs(got - ref)) <= bar
