"""The pixel passes (Eq. 10 / 13 over the disk, min / max, normalisation, polar
to pixels) at the places where their row spans, vector widths and groups can go
wrong, against the FP64 oracle.

Geometries sit on half pixels, so that FP32 and FP64 agree on which centres lie
in the disk.  Bars: sums of at most a few hundred FP32 terms per thread, so a
relative error below 512 * 2^-24 = 3.1e-5; min, max and count are exact; the
normalisation is three FP32 roundings of values up to |lo| + |hi|.  Polar to
pixels: theta N / 2 pi and the radial fraction carry a few FP32 roundings of
values up to N and N_rho, hence 8 * 2^-24 * max(N, N_rho) of a sample step; the
samples are within [-1, 1], so a step is at most 2 in each direction.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import grid, metrics, reconstruct as orc  # noqa: E402
from paper_2304_14492_gb300 import native as zm  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (h, w, geometry, column offset of the view, extra pitch): odd and tiny sizes,
# disks past the image's edge, wholly outside it and larger than it, rows on
# every 16-byte phase
SHAPES = [(1, 1, None, 0, 0), (3, 2, None, 1, 1), (33, 130, None, 0, 2), (70, 64, None, 0, 0), (257, 519, None, 3, 5),
          (64, 100, (20.0, 10.5, 40.0), 2, 0), (40, 40, (90.0, 20.0, 30.0), 0, 0), (31, 45, (22.0, 15.0, 200.0), 1, 2),
          (600, 1300, None, 0, 4)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2304_14492_gb300.build import build
    build()
    zm.lib()


def view(a, off, extra):
    h, w = a.shape
    buf = torch.zeros((h, w + off + extra), device=DEV)
    v = buf[:, off:off + w]
    v.copy_(torch.from_numpy(a))
    return v


def check_scores(row, f, g, count):
    assert row[3] == count
    if count == 0:
        assert np.isnan(row[0])
        return
    e1, mx = np.sum((f - g) ** 2) / np.sum(f ** 2), f.max()
    assert abs(row[0] - e1) <= 3.1e-5 * e1 and row[2] == mx
    e13 = np.sum((f - g) ** 2) / (mx * mx * count)
    assert abs(row[1] - e13) <= 3.1e-5 * e13


@pytest.mark.parametrize("h,w,geo,off,extra", SHAPES)
@pytest.mark.parametrize("same_phase", [True, False])
def test_disk_passes(h, w, geo, off, extra, same_phase):
    rng = np.random.default_rng(h * 1000 + w)
    f = rng.random((h, w), dtype=np.float32) + 0.25
    g = (f + 0.1 * rng.standard_normal((h, w))).astype(np.float32)
    mask = metrics.disk_mask(h, w, geo)
    fv, gv = view(f, off, extra), view(g, off if same_phase else off + 1, extra)
    plan = zm.zm_plan(4, 8, 16)
    try:
        err = torch.zeros((1, 4), device=DEV, dtype=torch.float64)
        mm = torch.zeros((1, 2), device=DEV)
        geos = None if geo is None else [geo]
        for _ in range(2):                                   # the second call finds the counter reset
            zm.zm_errors(plan, [fv], [gv], err, geometries=geos)
            zm.zm_disk_minmax(plan, [fv], mm, geometries=geos)
        target = torch.tensor([[-3.0, 255.0]], device=DEV)
        zm.zm_minmax_normalize(plan, [gv], target, geometries=geos)
        torch.cuda.synchronize()
    finally:
        zm.zm_plan_destroy(plan)
    check_scores(err[0].cpu().numpy(), f[mask].astype(np.float64), g[mask].astype(np.float64), mask.sum())
    lo, hi = mm[0].cpu().numpy()
    got = gv.cpu().numpy()
    assert np.array_equal(got[~mask], g[~mask])
    if mask.any():
        assert lo == f[mask].min() and hi == f[mask].max()
        ref = metrics.minmax_normalize(g.astype(np.float64), -3.0, 255.0, mask)
        assert np.max(np.abs(got[mask] - ref[mask])) <= 4 * 2.0 ** -24 * 258.0
    else:
        assert lo == np.inf and hi == -np.inf


def test_more_images_than_a_launch_takes():
    n = 131
    rng = np.random.default_rng(5)
    fs = rng.random((n, 13, 12 + 4), dtype=np.float32)
    widths = [9 + (b % 4) for b in range(n)]
    imgs = [torch.from_numpy(np.ascontiguousarray(fs[b][:, :widths[b]])).to(DEV) for b in range(n)]
    plan = zm.zm_plan(4, 8, 16)
    try:
        mm = torch.zeros((n, 2), device=DEV)
        zm.zm_disk_minmax(plan, imgs, mm)
        torch.cuda.synchronize()
    finally:
        zm.zm_plan_destroy(plan)
    for b in range(n):
        v = fs[b][:, :widths[b]][metrics.disk_mask(13, widths[b])]
        assert tuple(mm[b].cpu().numpy()) == (v.min(), v.max())


@pytest.mark.parametrize("n_rho,n_theta,batch,offset", [(1, 8, 1, 0), (9, 8, 3, 1), (130, 64, 2, 0), (37, 256, 2, 3)])
def test_polar_errors(n_rho, n_theta, batch, offset):
    rng = np.random.default_rng(n_rho)
    shape = (batch, n_rho, n_theta)
    f = rng.random(shape, dtype=np.float32) + 0.25
    g = (f + 0.1 * rng.standard_normal(shape)).astype(np.float32)
    fb, gb = (torch.zeros(f.size + 4, device=DEV) for _ in range(2))
    fd, gd = fb[:f.size].view(shape), gb[offset:offset + f.size].view(shape)
    fd.copy_(torch.from_numpy(f))
    gd.copy_(torch.from_numpy(g))
    err = torch.zeros((batch, 4), device=DEV, dtype=torch.float64)
    plan = zm.zm_plan(3, n_rho, n_theta)
    try:
        zm.zm_errors_polar(plan, fd, gd, batch, err)
        torch.cuda.synchronize()
    finally:
        zm.zm_plan_destroy(plan)
    for b in range(batch):
        check_scores(err[b].cpu().numpy(), f[b].astype(np.float64), g[b].astype(np.float64), n_rho * n_theta)


@pytest.mark.parametrize("gauss", [False, True])
@pytest.mark.parametrize("n_rho,n_theta", [(1, 8), (2, 16), (31, 64), (200, 32)])
def test_polar_to_pixels(n_rho, n_theta, gauss):
    sizes = [(60, 75)] * 5 + [(61, 75), (1, 1), (33, 36), (33, 36)]     # a group that is cut, and changes of size
    P = zm.zm_num_moments(3)
    rng = np.random.default_rng(n_rho)
    z = torch.from_numpy(rng.uniform(-0.05, 0.05, (len(sizes), P, 2)).astype(np.float32)).to(DEV)
    canv = [torch.full((h, w + 3), 7.0, device=DEV)[:, 1:1 + w] for h, w in sizes]
    polar = torch.empty((len(sizes), n_rho, n_theta), device=DEV)
    plan = zm.zm_plan(3, n_rho, n_theta, zm.ZM_GRID_GAUSS if gauss else 0)
    try:
        zm.zm_reconstruct_cartesian(plan, z, canv, polar, zm.ZM_NEUMANN)
        torch.cuda.synchronize()
    finally:
        zm.zm_plan_destroy(plan)
    rho, _ = grid.radial_nodes(n_rho, "gauss" if gauss else "midpoint")
    bar = 4 * 8 * 2.0 ** -24 * max(n_rho, n_theta, 8) * float(polar.abs().max())
    for b, (h, w) in enumerate(sizes):
        ref = orc.polar_to_cartesian(polar[b].double().cpu().numpy(), rho, h, w)
        got = canv[b].double().cpu().numpy()
        mask = metrics.disk_mask(h, w)
        assert np.all(got[~mask] == 0.0)
        assert np.max(np.abs(got - ref)) <= bar
