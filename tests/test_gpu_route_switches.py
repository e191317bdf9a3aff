"""Calls on both sides of the lines at which the default route changes (gather,
staged, tiles, by angles, samples an image and a call, image size, order and form): the same spectra and
moments as on plans told to stage or to tile, and the route told by its launches
(gathered and staged spectra are one kernel, tiles and ring FFT two; the staged
kernel alone builds a list, seen as nothing launched for it, and is told from the
gather by unaligned images, which only the gather takes).

All routes compute the same samples and transforms, so the comparison is exact.
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


def run(imgs, n_max, n_rho, n_theta, prec):
    """Moments, FP32 spectra and the launches of a warm call for each."""
    b = len(imgs)
    out = torch.empty((b, zm.zm_num_moments(n_max), 2), device=DEV)
    F = torch.empty((n_max + 1, b, 2, n_rho), device=DEV)
    n = []
    plan = zm.zm_plan(n_max, n_rho, n_theta, prec)
    try:
        for call in (lambda: zm.zm_moments(plan, imgs, out), lambda: zm.zm_ring_spectra(plan, imgs, F)):
            call()
            before = zm.zm_launch_count()
            call()
            n.append(zm.zm_launch_count() - before)
        zm.zm_plan_status(plan)
    finally:
        zm.zm_plan_destroy(plan)
    return out, F, n


# (side, n_max, n_rho, n_theta, batch, tiles for moments with blocks, tiles for FP32 rows)
CASES = [(128, 30, 64, 128, 3, False, False),
         (128, 30, 256, 256, 14, False, False), (128, 30, 256, 256, 15, False, False),  # 7/8 million: gathered, staged
         (128, 30, 256, 256, 24, False, False), (128, 30, 256, 256, 25, False, False),  # 1.5 million: staged, gathered
         (128, 65, 256, 256, 25, False, False), (128, 65, 256, 256, 41, False, False),  # order 65, 2.5 million: blocks staged, gathered
         (128, 30, 320, 256, 12, False, False),                                         # a grid above 2^16: gathered
         (1024, 30, 256, 256, 32, False, False), (1024, 30, 256, 256, 33, True, True),  # large images, 2 million: gathered, tiles
         (128, 30, 256, 512, 4, False, False), (128, 30, 256, 512, 5, False, False),    # blocks, half a million: gathered, staged
         (128, 30, 256, 512, 12, False, False), (128, 30, 256, 512, 13, False, False),  # FP32 rows, 1.5 million: gathered, staged
         (400, 30, 64, 512, 17, False, False),                                          # large images, blocks: gathered
         (128, 30, 257, 512, 1, True, True),                                            # a grid above 2^17: tiles
         (128, 30, 128, 1024, 12, False, False), (128, 30, 128, 1024, 13, False, False),  # 1.5 million: gathered, staged
         (128, 30, 129, 1024, 7, False, False), (128, 30, 256, 1024, 4, False, True),   # a million: FP32 rows by tiles
         (128, 30, 256, 1024, 5, False, True), (128, 30, 256, 1024, 6, True, True),     # 1.25 million: tiles
         (128, 30, 16, 2048, 1, False, False), (128, 30, 65, 2048, 1, True, True)]      # 2048: staged, tiles


@pytest.mark.parametrize("side,n_max,n_rho,n_theta,batch,tiles_blk,tiles_f32", CASES)
def test_both_sides_of_every_line(side, n_max, n_rho, n_theta, batch, tiles_blk, tiles_f32, monkeypatch):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(n_rho * n_theta + batch)
    imgs = [torch.rand((side, side), device=DEV, generator=gen) for _ in range(batch)]
    out, F, n = run(imgs, n_max, n_rho, n_theta, zm.ZM_PREC_BF16X3)
    assert n == [3 if tiles_blk else 2, 2 if tiles_f32 else 1]
    _, F32, n32 = run(imgs, n_max, n_rho, n_theta, zm.ZM_PREC_FP32)
    assert n32 == [3 if tiles_f32 else 2, 2 if tiles_f32 else 1]     # by the form of the spectra, not the plan
    assert torch.equal(F, F32)
    for mode in ("0", "1"):
        monkeypatch.setenv("ZM_FUSED", mode)
        told, Ft, nt = run(imgs, n_max, n_rho, n_theta, zm.ZM_PREC_BF16X3)
        if mode == "0":
            assert nt == [3, 2]
        assert torch.equal(told, out) and torch.equal(Ft, F)
    monkeypatch.delenv("ZM_FUSED")
    odd = [torch.zeros((side, side + 1), device=DEV)[:, :side] for _ in imgs]
    for o, i in zip(odd, imgs):
        o.copy_(i)
    told, Ft, _ = run(odd, n_max, n_rho, n_theta, zm.ZM_PREC_BF16X3)
    assert torch.equal(told, out) and torch.equal(Ft, F)
