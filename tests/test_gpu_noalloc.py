"""zm_project_noalloc against the radial sum in 64 bits, for every image of a batch
and on plans of every precision (the call computes in FP32 whatever the plan), up to
the largest batch it takes; the next one is refused.

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


def largest_batch(n_max):
    return (1 << 21) // (2 * zm.zm_num_moments(n_max))


@pytest.mark.parametrize("prec", ["FP32", "BF16X3", "FP16X3"])
@pytest.mark.parametrize("n_max,n_rho,n_theta,batch", [(50, 256, 256, 7), (200, 64, 512, None)])
def test_every_image_matches_the_sum_in_64_bits(prec, n_max, n_rho, n_theta, batch):
    batch = batch or largest_batch(n_max)
    F = np.random.default_rng(n_max + batch).standard_normal((n_max + 1, batch, 2, n_rho)).astype(np.float32)
    Fd = torch.from_numpy(F).to(DEV)
    P = zm.zm_num_moments(n_max)
    out = torch.full((batch, P, 2), float("nan"), device=DEV)
    table = torch.empty((P, n_rho), device=DEV, dtype=torch.float64)
    wr = torch.empty(n_rho, device=DEV, dtype=torch.float64)
    plan = zm.zm_plan(n_max, n_rho, n_theta, getattr(zm, "ZM_PREC_" + prec))
    try:
        zm.zm_project_noalloc(plan, Fd, batch, out, zm.ZM_NEUMANN)
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
            f = 0.5 if m == 0 else 1.0
            ref = f * (F[m].astype(np.float64) @ a)
            bar = (n_rho + 2) * 2.0 ** -24 * f * (np.abs(F[m]).astype(np.float64) @ np.abs(a))
            assert np.all(np.abs(got[:, k] - ref) <= bar), (n, m)


def test_one_image_more_than_the_largest_batch_is_refused():
    n_max, n_rho, n_theta = 200, 8, 512
    batch = largest_batch(n_max) + 1
    out = torch.zeros((batch, zm.zm_num_moments(n_max), 2), device=DEV)
    plan = zm.zm_plan(n_max, n_rho, n_theta, zm.ZM_PREC_FP32)
    try:
        with pytest.raises(zm.ZmError) as e:
            zm.zm_project_noalloc(plan, torch.zeros((n_max + 1, batch, 2, n_rho), device=DEV), batch, out)
        assert e.value.status == zm.ZM_EINVAL
    finally:
        zm.zm_plan_destroy(plan)
