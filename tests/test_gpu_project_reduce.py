"""The slices' sums of the tensor-core projection (zm_project on bf16x3 and fp16x3
plans) at the edges of the row to moment map: every parity of n_max, batches that
divide no warp or block, one slice and many, with and without the Neumann factor.

Bar per moment: the split's 3 * 2^-16 (bf16 halves: 2^-8 of 2^-8) or 3 * 2^-22 (fp16)
plus FP32 accumulation (n_rho + 8) 2^-24, of S_nm = sum_i |a_i f_i|, and 2^-38 of
a_max sum |f| + f_max sum |a| for halves below fp16's range.
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


@pytest.mark.parametrize("prec,split", [(zm.ZM_PREC_BF16X3, 3 * 2.0 ** -16), (zm.ZM_PREC_FP16X3, 3 * 2.0 ** -22)])
@pytest.mark.parametrize("n_max,n_rho,n_theta", [(0, 5, 8), (1, 64, 8), (2, 65, 8), (3, 640, 8), (31, 128, 64), (64, 130, 256),
                                                 (130, 70, 512)])
@pytest.mark.parametrize("batch,flags", [(1, 0), (3, zm.ZM_NEUMANN), (65, zm.ZM_NEUMANN), (257, 0)])
def test_every_moment_in_its_place(n_max, n_rho, n_theta, batch, flags, prec, split):
    rng = np.random.default_rng(n_max * 1000 + batch)
    F = rng.standard_normal((n_max + 1, batch, 2, n_rho)).astype(np.float32)
    P = zm.zm_num_moments(n_max)
    out = torch.full((batch, P, 2), float("nan"), device=DEV)
    table = torch.empty((P, n_rho), device=DEV, dtype=torch.float64)
    wr = torch.empty(n_rho, device=DEV, dtype=torch.float64)
    plan = zm.zm_plan(n_max, n_rho, n_theta, prec)
    try:
        zm.zm_project(plan, torch.from_numpy(F).to(DEV), batch, out, flags)
        zm.zm_plan_table(plan, table)
        zm.zm_plan_nodes(plan, None, wr)
        zm.zm_plan_status(plan)
    finally:
        zm.zm_plan_destroy(plan)
    got, R, w = out.cpu().numpy().astype(np.float64), table.cpu().numpy(), wr.cpu().numpy()
    nms = [(n, m) for n in range(n_max + 1) for m in range(n % 2, n + 1, 2)]
    A = np.stack([2.0 * (n + 1) / n_theta * w * R[zm.zm_index(n, m)] for n, m in nms])
    for k, (n, m) in enumerate(nms):
        f = F[m].astype(np.float64)
        eps = 0.5 if flags and m == 0 else 1.0
        S = np.abs(f) @ np.abs(A[k])
        low = np.abs(A).max() * np.abs(f).sum(axis=2) + np.abs(f).max(axis=2) * np.abs(A[k]).sum()
        bar = (split + (n_rho + 8) * 2.0 ** -24) * S + 2.0 ** -38 * low
        assert np.all(np.abs(got[:, zm.zm_index(n, m)] - eps * (f @ A[k])) <= bar), (n, m)
