"""The Cartesian sums at the edges of their 32 x 16 tiles of point pairs, for
every residue of m mod 4, and at recurrence lengths up to several hundred steps.

Bar: |R_nm| <= 1, so the moment's scale is (n + 1) / (pi r^2) sum |f|; a step of
the recurrence rounds twice and carries a rounded coefficient (3 * 2^-24 of a
value of about 1), an error that the recurrence passes on about unchanged on
[0, 1], and the angular factor takes 2 log2(m) roundings: 8 (s + 1 + log2(m + 1))
2^-24 of the scale, s = (n - m) / 2.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import cartesian as ocart, grid  # noqa: E402
from paper_2304_14492_gb300 import native as zm  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
PAIRS = [(0, 0), (1, 1), (2, 2), (3, 3), (4, 4), (60, 2), (61, 3), (400, 2), (399, 101)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2304_14492_gb300.build import build
    build()
    zm.lib()


@pytest.mark.parametrize("h,w,geo", [
    (2, 2, None), (3, 3, None), (32, 32, None), (33, 33, None), (62, 62, None), (65, 65, None), (128, 130, None),
    (31, 33, (16.25, 14.0, 15.5)), (65, 64, (31.0, 30.5, 34.0)), (70, 70, (34.5, 30.5, 50.0))])
def test_tiles_orders_and_counts(h, w, geo):
    rng = np.random.default_rng(h * 100 + w)
    imgs = [rng.random((h, w), dtype=np.float32) for _ in range(2)]
    g = geo if geo else grid.default_geometry(h, w)
    for count in (1, 2, 3, len(PAIRS)):                     # one, two and four pairs per pass
        pairs = PAIRS[-count:]
        out = torch.full((2, count, 2), float("nan"), device=DEV)
        work = torch.empty(zm.zm_cartesian_work_bytes(2, count) // 8 + 1, dtype=torch.float64, device=DEV)
        ts = [torch.from_numpy(i).to(DEV) for i in imgs]
        zm.zm_cartesian_moments(ts, pairs, out, work, 0, geometries=[geo] * 2 if geo else None)
        torch.cuda.synchronize()
        got = out.double().cpu().numpy()
        for b, img in enumerate(imgs):
            ref = ocart.moments_cartesian(img, pairs, g)
            rows, cols, _, _ = ocart.disk_pixels(h, w, g)
            total = np.sum(np.abs(img[rows, cols]).astype(np.float64))
            for k, (n, m) in enumerate(pairs):
                bar = 8 * ((n - m) // 2 + 1 + np.log2(m + 1)) * 2.0 ** -24 * (n + 1) / (np.pi * g[2] ** 2) * total
                z = got[b, k, 0] + 1j * got[b, k, 1]
                assert abs(z - ref[k]) <= bar, (n, m, z, ref[k], bar)
