"""fp16x3 projection of given spectra whose columns, orders and radial slices
differ by many powers of two, and whose rows start on any 4-byte boundary.

Bar per moment: the split's 3 * 2^-22 plus FP32 accumulation (n_rho + 8) 2^-24,
of S_nm = sum_i |a_i f_i|, and 2^-30 of the column's largest S of that m for
weights below fp16's range.
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


@pytest.mark.parametrize("n_max,n_rho,n_theta,batch,offset", [(20, 64, 64, 1, 0), (30, 200, 64, 9, 0), (30, 201, 64, 3, 1),
                                                              (12, 256, 32, 70, 1), (60, 68, 128, 2, 2)])
def test_scales(n_max, n_rho, n_theta, batch, offset):
    rng = np.random.default_rng(n_rho + batch)
    F = rng.standard_normal((n_max + 1, batch, 2, n_rho))
    F *= 2.0 ** rng.integers(-30, 31, (n_max + 1, batch, 2, 1))          # per order and column
    F[..., n_rho // 2:] *= 2.0 ** 12                                     # per slice of the radius
    F = F.astype(np.float32)
    buf = torch.zeros(F.size + 4, device=DEV)
    Fd = buf[offset:offset + F.size].view(F.shape)
    Fd.copy_(torch.from_numpy(F))
    P = zm.zm_num_moments(n_max)
    out = torch.full((batch, P, 2), float("nan"), device=DEV)
    table = torch.empty((P, n_rho), device=DEV, dtype=torch.float64)
    wr = torch.empty(n_rho, device=DEV, dtype=torch.float64)
    plan = zm.zm_plan(n_max, n_rho, n_theta, zm.ZM_PREC_FP16X3)
    try:
        zm.zm_project(plan, Fd, batch, out, 0)
        zm.zm_plan_table(plan, table)
        zm.zm_plan_nodes(plan, None, wr)
        zm.zm_plan_status(plan)
    finally:
        zm.zm_plan_destroy(plan)
    got, R, w = out.cpu().numpy().astype(np.float64), table.cpu().numpy(), wr.cpu().numpy()
    for m in range(n_max + 1):
        ns = list(range(m, n_max + 1, 2))
        a = np.stack([2.0 * (n + 1) / n_theta * w * R[zm.zm_index(n, m)] for n in ns])
        f = F[m].astype(np.float64)
        ref, S = f @ a.T, np.abs(f) @ np.abs(a).T                        # [batch][2][order]
        bar = (3 * 2.0 ** -22 + (n_rho + 8) * 2.0 ** -24) * S + 2.0 ** -30 * S.max(axis=2, keepdims=True)
        z = got[:, [zm.zm_index(n, m) for n in ns], :].transpose(0, 2, 1)
        assert np.all(np.abs(z - ref) <= bar), m
