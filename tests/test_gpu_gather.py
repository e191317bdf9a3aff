"""The gather kernel against the staged and tiled ones and the general sampling
path, bit for bit, over every ring length it is built for: rings wholly inside
the image (no bounds tests), rings at its edge, outside it, tiny and unaligned
images, strided rows, FP32 spectra and operand blocks.

All paths interpolate with the same float operations, so the polar samples of
zm_moments_ex, and the moments, are equal to those of a plan that may not gather
(ZM_FUSED=0, aligned images) and to the same image seen through an unaligned
view; zm_resample of an unaligned view takes the general sampling code.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import moments as om  # noqa: E402
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


GEOMETRIES = [None, (30.0, 21.5, 18.0), (0.0, 0.0, 25.0), (63.5, 40.0, 60.0), (200.0, 200.0, 40.0)]


@pytest.mark.parametrize("n_max,n_rho,n_theta", [(3, 5, 8), (5, 9, 16), (9, 40, 32), (20, 33, 64), (40, 66, 128),
                                                 (60, 70, 256), (100, 64, 512), (150, 40, 1024), (300, 16, 2048)])
@pytest.mark.parametrize("prec", [zm.ZM_PREC_FP32, zm.ZM_PREC_BF16X3])
def test_paths_agree(monkeypatch, n_max, n_rho, n_theta, prec):
    rng = np.random.default_rng(n_theta + n_rho)
    a = rng.random((64, 80), dtype=np.float32)
    P = zm.zm_num_moments(n_max)
    aligned = torch.from_numpy(a).to(DEV)
    odd = torch.zeros((64, 83), device=DEV)[:, 1:81]
    odd.copy_(aligned)
    got = {}
    for name, env, img in (("auto", None, aligned), ("odd", None, odd), ("two-pass", "0", aligned)):
        if env is None:
            monkeypatch.delenv("ZM_FUSED", raising=False)
        else:
            monkeypatch.setenv("ZM_FUSED", env)
        plan = zm.zm_plan(n_max, n_rho, n_theta, prec)
        try:
            geos = GEOMETRIES + [None]
            n = len(geos)
            out = torch.full((n, P, 2), float("nan"), device=DEV)
            out_ex = torch.full((n, P, 2), float("nan"), device=DEV)
            fh = torch.full((n, n_rho, n_theta), float("nan"), device=DEV)
            fr = torch.full((n, n_rho, n_theta), float("nan"), device=DEV)
            zm.zm_moments(plan, [img] * n, out, 0, geometries=geos)
            zm.zm_moments_ex(plan, [img] * n, out_ex, fh, 0, geometries=geos)
            zm.zm_resample(plan, [img] * n, fr, geometries=geos)
            zm.zm_plan_status(plan)
            assert torch.equal(out, out_ex) and torch.equal(fh, fr)
            got[name] = (out, fh)
        finally:
            zm.zm_plan_destroy(plan)
    for name in ("odd", "two-pass"):
        assert torch.equal(got["auto"][1], got[name][1]), name
        assert torch.equal(got["auto"][0], got[name][0]), name
    for b in (0, 1, 3):
        ref = om.moments(a.astype(np.float64), n_max, n_rho, n_theta, geometry=GEOMETRIES[b])
        z = got["auto"][0][b].double().cpu().numpy()
        assert np.max(np.abs(z[:, 0] + 1j * z[:, 1] - ref)) <= 1e-4 * np.max(np.abs(ref))
