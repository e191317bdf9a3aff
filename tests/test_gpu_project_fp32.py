"""The FP32 projection kernel on given spectra at the edges of its tiles (orders,
columns, node chunks, unaligned operands), against the radial sum in 64 bits.

Bar per moment: every product carries the rounding of the FP32 weight and of one
fused multiply-add, and a sum of n_rho terms in any order adds at most n_rho
roundings: (n_rho + 2) 2^-24 S_nm with S_nm = sum_i |a_i f_i| (re and im apart).
"""

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


@pytest.mark.parametrize("n_max,n_rho,n_theta,batch,offset", [
    (0, 1, 8, 1, 0), (1, 9, 8, 4, 0), (20, 32, 64, 1, 0), (20, 37, 64, 5, 0), (63, 64, 128, 8, 0), (64, 501, 256, 9, 0),
    (130, 260, 512, 16, 0), (130, 260, 512, 17, 1), (200, 96, 512, 3, 2), (7, 1024, 16, 40, 0)])
@pytest.mark.parametrize("neumann", [False, True])
def test_projection_of_given_spectra(n_max, n_rho, n_theta, batch, offset, neumann):
    rng = np.random.default_rng(n_max * 100 + batch)
    F = rng.standard_normal((n_max + 1, batch, 2, n_rho)).astype(np.float32)
    buf = torch.zeros(F.size + 4, device=DEV)
    Fd = buf[offset:offset + F.size].view(F.shape)
    Fd.copy_(torch.from_numpy(F))
    P = zm.zm_num_moments(n_max)
    out = torch.full((batch, P, 2), float("nan"), device=DEV)
    table = torch.empty((P, n_rho), device=DEV, dtype=torch.float64)
    wr = torch.empty(n_rho, device=DEV, dtype=torch.float64)
    plan = zm.zm_plan(n_max, n_rho, n_theta, zm.ZM_PREC_FP32)
    try:
        zm.zm_project(plan, Fd, batch, out, zm.ZM_NEUMANN if neumann else 0)
        zm.zm_plan_table(plan, table)
        zm.zm_plan_nodes(plan, None, wr)
        torch.cuda.synchronize()
    finally:
        zm.zm_plan_destroy(plan)
    got, R, w = out.cpu().numpy().astype(np.float64), table.cpu().numpy(), wr.cpu().numpy()
    for n in range(n_max + 1):
        for m in range(n % 2, n + 1, 2):
            k = zm.zm_index(n, m)
            a = 2.0 * (n + 1) / n_theta * w * R[k]
            f = 0.5 if neumann and m == 0 else 1.0
            ref = f * (F[m].astype(np.float64) @ a)
            bar = (n_rho + 2) * 2.0 ** -24 * f * (np.abs(F[m]).astype(np.float64) @ np.abs(a))
            assert np.all(np.abs(got[:, k] - ref) <= bar), (n, m)
