"""The ring FFT into operand blocks with one, two and four images to an item, from
given polar samples: batches that leave an item's images partly absent and blocks
past the last ring, against the oracle and against each image alone.

A ring's spectrum depends on that ring alone, and the projection sums an image's
columns alone, so an image gives the same moments, bit for bit, in any batch that
takes the same projection form; other batches agree to the split's bar.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import metrics, moments as om  # noqa: E402
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


@pytest.mark.parametrize("n_max,n_rho,n_theta", [(3, 7, 8), (10, 65, 32), (40, 130, 128), (100, 72, 512), (120, 200, 1024),
                                                 (200, 9, 2048)])
@pytest.mark.parametrize("batch", [1, 2, 3, 5, 8, 37])
def test_batches(n_max, n_rho, n_theta, batch):
    rng = np.random.default_rng(n_rho + batch)
    f = rng.random((batch, n_rho, n_theta), dtype=np.float32)
    fd = torch.from_numpy(f).to(DEV)
    P = zm.zm_num_moments(n_max)
    out = torch.full((batch, P, 2), float("nan"), device=DEV)
    one = torch.full((1, P, 2), float("nan"), device=DEV)
    plan = zm.zm_plan(n_max, n_rho, n_theta, zm.ZM_PREC_BF16X3)
    try:
        zm.zm_moments_polar(plan, fd, batch, out)
        zm.zm_plan_status(plan)
        got = out.double().cpu().numpy()
        for b in sorted({0, batch // 2, batch - 1}):
            ref = om.moments_polar(f[b].astype(np.float64), n_max)
            z = got[b, :, 0] + 1j * got[b, :, 1]
            assert metrics.rel_max_err(z, ref) <= 2e-5, b
            zm.zm_moments_polar(plan, fd[b:b + 1].contiguous(), 1, one)
            zm.zm_plan_status(plan)
            alone = one.double().cpu().numpy()[0]
            assert metrics.rel_max_err(alone[:, 0] + 1j * alone[:, 1], z) <= 1e-6, b
    finally:
        zm.zm_plan_destroy(plan)
