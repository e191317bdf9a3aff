"""fp16x3 moments where some orders have radial slices of vanishing spectra:
smooth images on a zero background, whose rings fall off below FP32's normal
range, and given spectra with such slices beside ordinary ones.

Bars.  Images: the split form's 2e-5 of the largest moment, against the 64-bit
oracle.  Spectra, per moment: the split's 3 * 2^-22 plus FP32 accumulation
(n_rho + 8) 2^-24 of S_nm = sum_i |a_i f_i|; what the halves lose below fp16's
range, 2^-25 of a scaled operand: the plan's weights are scaled to a largest one
of 2^13 or more (2^-38 a_max sum_i |f_i|) and so are the spectra (2^-38 f_max
sum_i |a_i|); and n_rho 2^-126 for slices that the scale cannot lift (scaled by
2^126 over the weights' scale, of which a half below 2^-14 may be lost: n_rho
2^14 2^-14 2^-126).
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


@pytest.mark.parametrize("side,sigma,dx,dy,n_rho,n_theta", [(512, 16.0, 0.0, 0.0, 256, 256),
                                                           (1024, 20.0, 61.0, -40.0, 512, 512)])
def test_gaussian_on_a_zero_background(side, sigma, dx, dy, n_rho, n_theta):
    n_max = 80
    c = (side - 1) / 2.0
    y, x = np.mgrid[0:side, 0:side].astype(np.float32)
    img = np.exp(-((x - np.float32(c + dx)) ** 2 + (y - np.float32(c + dy)) ** 2) / np.float32(2.0 * sigma * sigma))
    assert img.dtype == np.float32 and img.max() > 0.9 and (img == 0.0).any()
    out = torch.full((1, zm.zm_num_moments(n_max), 2), float("nan"), device=DEV)
    plan = zm.zm_plan(n_max, n_rho, n_theta, zm.ZM_PREC_FP16X3)
    try:
        zm.zm_moments(plan, [torch.from_numpy(img).to(DEV)], out)
        zm.zm_plan_status(plan)
    finally:
        zm.zm_plan_destroy(plan)
    o = out[0].double().cpu().numpy()
    assert np.isfinite(o).all()
    ref = om.moments(img.astype(np.float64), n_max, n_rho, n_theta)
    assert metrics.rel_max_err(o[:, 0] + 1j * o[:, 1], ref) <= 2e-5


@pytest.mark.parametrize("n_max,n_rho,n_theta,batch", [(30, 320, 64, 3), (80, 319, 256, 1), (12, 1024, 32, 70)])
def test_vanishing_slices_beside_ordinary_ones(n_max, n_rho, n_theta, batch):
    rng = np.random.default_rng(n_rho)
    F = rng.standard_normal((n_max + 1, batch, 2, n_rho))
    powers = np.array([0, -100, -116, -126, -140])
    for c in range(0, n_rho, 64):                            # the kernel's slices are runs of 64 nodes
        F[..., c:c + 64] *= 2.0 ** powers[(c // 64 + np.arange(n_max + 1)) % 5][:, None, None, None]
    F[:, :, 1] *= 2.0 ** -113                                # every imaginary part below the range as a whole
    F[..., ::3] = 0.0
    F = F.astype(np.float32)
    Fd = torch.from_numpy(F).to(DEV)
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
    assert np.isfinite(got).all()
    a_max = max(2.0 * (n + 1) / n_theta * np.abs(w * R[zm.zm_index(n, m)]).max()
                for n in range(n_max + 1) for m in range(n % 2, n + 1, 2))
    for m in range(n_max + 1):
        ns = list(range(m, n_max + 1, 2))
        a = np.stack([2.0 * (n + 1) / n_theta * w * R[zm.zm_index(n, m)] for n in ns])
        f = F[m].astype(np.float64)
        ref, S = f @ a.T, np.abs(f) @ np.abs(a).T                        # [batch][2][order]
        low = a_max * np.abs(f).sum(axis=2)[..., None] + np.abs(f).max(axis=2)[..., None] * np.abs(a).sum(axis=1)
        bar = (3 * 2.0 ** -22 + (n_rho + 8) * 2.0 ** -24) * S + 2.0 ** -38 * low
        z = got[:, [zm.zm_index(n, m) for n in ns], :].transpose(0, 2, 1)
        assert np.all(np.abs(z - ref) <= bar + n_rho * 2.0 ** -126), m
