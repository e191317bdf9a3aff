"""The FP32 radial reconstruction of larger batches, at the edges of its
node tiles (256 nodes, 128 where rows are not 16-byte aligned), ring blocks, image
groups of 16 and chunks of eight orders, through zm_reconstruct, against the oracle;
an image alone, which takes the other kernel, agrees.

Bar per sample: |R_nm| <= 1, so with Sigma = sum c_m |Z_nm| the table's rounding,
chunks of 8 fused steps and K_m / 8 <= 9 additions, and the inverse FFT (a few
roundings per butterfly stage, at most 11 stages) stay below 128 * 2^-24 Sigma.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import reconstruct as orc  # noqa: E402
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


@pytest.mark.parametrize("n_max,n_rho,n_theta", [(0, 1, 8), (3, 4, 8), (14, 64, 32), (15, 63, 32), (17, 65, 64), (30, 127, 64),
                                                 (31, 256, 64), (63, 129, 128), (130, 260, 512), (127, 257, 256)])
@pytest.mark.parametrize("batch", [5, 8, 16, 17, 35])
@pytest.mark.parametrize("prec", [zm.ZM_PREC_FP32, zm.ZM_PREC_FP16X3])
def test_radial_wide(n_max, n_rho, n_theta, batch, prec):
    rng = np.random.default_rng(n_rho * 100 + batch)
    P = zm.zm_num_moments(n_max)
    z = rng.standard_normal((batch, P, 2)).astype(np.float32)
    zd = torch.from_numpy(z).to(DEV)
    out = torch.full((batch, n_rho, n_theta), float("nan"), device=DEV)
    one = torch.full((1, n_rho, n_theta), float("nan"), device=DEV)
    plan = zm.zm_plan(n_max, n_rho, n_theta, prec)
    try:
        zm.zm_reconstruct(plan, zd, batch, out, zm.ZM_NEUMANN)
        zm.zm_reconstruct(plan, zd[batch - 1:], 1, one, zm.ZM_NEUMANN)
        torch.cuda.synchronize()
    finally:
        zm.zm_plan_destroy(plan)
    got = out.double().cpu().numpy()
    sigma = 2.0 * np.sum(np.hypot(z[..., 0].astype(np.float64), z[..., 1]), axis=1)
    for b in sorted({0, 1, 4, batch // 2, batch - 2, batch - 1}):
        Z = z[b, :, 0].astype(np.float64) + 1j * z[b, :, 1]
        ref = orc.reconstruct_polar(Z, n_max, n_rho, n_theta, neumann=True)
        assert np.max(np.abs(got[b] - ref)) <= 128 * 2.0 ** -24 * sigma[b], b
    assert np.isfinite(got).all()
    alone = one[0].double().cpu().numpy()
    assert np.max(np.abs(alone - got[-1])) <= 256 * 2.0 ** -24 * sigma[-1]
