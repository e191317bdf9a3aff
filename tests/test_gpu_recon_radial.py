"""The FP32 radial reconstruction at the edges of its node tiles, image groups
and warps, through zm_reconstruct, against the oracle.

Bar per sample: |R_nm| <= 1, so with Sigma = sum c_m |Z_nm| the table's rounding,
K_m <= 66 fused steps in any order and the inverse FFT (a few roundings per
butterfly stage, at most 11 stages) stay below 128 * 2^-24 Sigma.
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


@pytest.mark.parametrize("n_max,n_rho,n_theta", [(0, 1, 8), (7, 33, 16), (20, 128, 64), (63, 130, 128), (130, 260, 512)])
@pytest.mark.parametrize("batch", [1, 2, 3, 5, 9])
def test_radial(n_max, n_rho, n_theta, batch):
    rng = np.random.default_rng(n_rho * 10 + batch)
    P = zm.zm_num_moments(n_max)
    z = rng.standard_normal((batch, P, 2)).astype(np.float32)
    out = torch.full((batch, n_rho, n_theta), float("nan"), device=DEV)
    plan = zm.zm_plan(n_max, n_rho, n_theta, zm.ZM_PREC_FP32)
    try:
        zm.zm_reconstruct(plan, torch.from_numpy(z).to(DEV), batch, out, zm.ZM_NEUMANN)
        torch.cuda.synchronize()
    finally:
        zm.zm_plan_destroy(plan)
    got = out.double().cpu().numpy()
    for b in range(batch):
        Z = z[b, :, 0].astype(np.float64) + 1j * z[b, :, 1]
        ref = orc.reconstruct_polar(Z, n_max, n_rho, n_theta, neumann=True)
        assert np.max(np.abs(got[b] - ref)) <= 128 * 2.0 ** -24 * 2.0 * np.sum(np.abs(Z))
