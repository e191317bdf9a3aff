"""The workloads whose time counts: Zernike moments, reconstruction, colour
frames, Cartesian sums, uneven batches and uploads, each through the entry
points a program calls, over the sizes this library is used at.

A case is a dict of plain values.  ``kind`` says which entry points run:

  moments   zm_moments on a batch of device images of one size
  errors    zm_reconstruct_errors (decode on the polar nodes, score against the
            stored polar samples)
  recon     zm_reconstruct (decode on the polar nodes)
  colour    decode a frame's bands onto pixels: zm_disk_minmax of the originals,
            zm_reconstruct_cartesian, zm_minmax_normalize, zm_errors
  cartesian zm_cartesian_moments (chosen moments summed over the pixels)
  uneven    zm_batch_run: requests of mixed sizes, orders and grids
  upload    zm_upload_disk of pinned host frames, then zm_moments

``prepare`` makes what a program holds before the call (images or moments on
the device, the plan, descriptor arrays, output buffers); ``run`` is one pass.
``exact`` gives the same results from the formulas in 64 bits with torch alone.
"""

import math

import numpy as np
import torch

from paper_2304_14492_gb300 import native as zm

PREC = {"fp32": zm.ZM_PREC_FP32, "bf16x3": zm.ZM_PREC_BF16X3, "fp16x3": zm.ZM_PREC_FP16X3}


def _case(name, kind, h, w, batch, n_max, n_rho, n_theta, prec="bf16x3", gauss=False, neumann=False, **more):
    c = {"kind": kind, "h": h, "w": w, "batch": batch, "n_max": n_max, "n_rho": n_rho, "n_theta": n_theta,
         "prec": prec, "gauss": gauss, "neumann": neumann, "blobs": 8}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one thumbnail, every moment to order 20: the smallest call, all latency
        _case("moments_64_fp32", "moments", 64, 64, 1, 20, 32, 64, prec="fp32", blobs=3),
        # a small batch of photographs at a moderate order (descriptors for matching)
        _case("moments_512_b16", "moments", 512, 512, 16, 50, 256, 256),
        # one video frame as it arrives: the latency of a camera loop
        _case("moments_4k_b1", "moments", 2160, 3840, 1, 100, 1024, 1024, blobs=32),
        # 4K frames in batches, the headline throughput workload
        _case("moments_4k_b16", "moments", 2160, 3840, 16, 100, 1024, 1024, blobs=32),
        # high orders on Gauss-Legendre nodes in plain FP32: the accuracy mode
        _case("moments_1024_n200_fp32", "moments", 1024, 1024, 16, 200, 512, 512, prec="fp32", gauss=True, blobs=16),
        # crops of a larger image: odd sizes, unaligned rows, an off-centre disk
        _case("moments_crop_fp16", "moments", 1001, 1503, 5, 80, 501, 256, prec="fp16x3", neumann=True, crop=True),
        # decode and score a batch of 4K frames on the polar grid (Eq. 9, 10, 13)
        _case("errors_4k_b16", "errors", 0, 0, 16, 100, 1024, 1024, neumann=True),
        # decode at very high order, FP32, Gauss-Legendre nodes (the stability study)
        _case("recon_n500_fp32", "recon", 0, 0, 4, 500, 512, 1024, prec="fp32", gauss=True, neumann=True),
        # decode one 4K colour frame onto its pixels, normalise and score its bands
        _case("colour_4k", "colour", 2160, 3840, 3, 100, 1024, 1024, neumann=True, blobs=32),
        # one moment of one large square frame by summation over its pixels
        _case("cartesian_4000", "cartesian", 4000, 4000, 1, 100, 0, 0, prec="fp32", pairs="100:36", blobs=24),
        # a mixed batch of requests replayed as one graph
        _case("uneven_256", "uneven", 0, 0, 256, 80, 0, 0, spec=3),
        # frames still on the host: pinned frames in, moments out
        _case("upload_4k_b8", "upload", 2160, 3840, 8, 100, 1024, 1024, blobs=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _theta(n_max):
    t = 8
    while t < 2 * n_max + 2:
        t *= 2
    return t


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["moments"] * 6 + ["errors", "recon", "colour", "cartesian", "uneven", "upload"])
    prec = rng.choice(["bf16x3", "bf16x3", "fp32", "fp16x3"])
    gauss, neumann = rng.random() < 0.25, rng.random() < 0.5
    n_max = _log(rng, 4, 200)
    n_theta = min(2048, _theta(n_max) * rng.choice([1, 1, 2, 4]))
    if kind == "moments":
        h, w = _log(rng, 33, 2160), _log(rng, 33, 3840)
        if rng.random() < 0.4:
            h, w = (h + 3) // 4 * 4, (w + 3) // 4 * 4
        if rng.random() < 0.3:
            w = h
        batch = max(1, min(_log(rng, 1, 32), 60_000_000 // (h * w)))
        n_rho = max(8, min(1024, int(min(h, w) * rng.uniform(0.4, 0.6))))
        return _case(None, kind, h, w, batch, n_max, n_rho, min(n_theta, 1024), prec, gauss, neumann,
                     crop=rng.random() < 0.3)
    if kind == "errors":
        return _case(None, kind, 0, 0, _log(rng, 1, 16), min(n_max, 150), _log(rng, 32, 1024), min(n_theta, 1024),
                     prec, gauss, neumann)
    if kind == "recon":
        n_max = _log(rng, 8, 500)
        return _case(None, kind, 0, 0, _log(rng, 1, 8), n_max, max(16, min(512, n_max + _log(rng, 2, 300))),
                     min(1024, max(n_theta, _theta(n_max))), prec, gauss, neumann)
    if kind == "colour":
        h = _log(rng, 120, 2160)
        w = min(3840, int(h * rng.uniform(1.0, 1.8)))
        return _case(None, kind, h, w, 3, min(n_max, 100), max(16, h // 2 if h < 2000 else 1024),
                     min(n_theta, 1024), prec, gauss, neumann)
    if kind == "cartesian":
        side = _log(rng, 128, 4000)
        pairs = []
        for _ in range(1 if side > 2500 else rng.randint(1, 6)):
            n = _log(rng, 2, 100 if side > 2500 else 200)
            pairs.append("%d:%d" % (n, rng.randrange(n % 2, n + 1, 2)))
        return _case(None, kind, side, side, 1 if side > 1000 else rng.randint(1, 8), 200, 0, 0, "fp32", False, neumann,
                     pairs=",".join(pairs))
    if kind == "uneven":
        return _case(None, kind, 0, 0, _log(rng, 8, 200), 80, 0, 0, prec, gauss, neumann, spec=rng.randrange(10**6))
    h = _log(rng, 240, 2160)
    w = min(3840, int(h * rng.uniform(1.0, 1.8)) // 4 * 4)
    return _case(None, kind, h, w, max(1, min(_log(rng, 1, 16), 60_000_000 // (h * w))), min(n_max, 100),
                 max(16, min(1024, h // 2)), min(n_theta, 1024), prec, gauss, neumann)


# ------------------------------------------------------------------ inputs
def _frame(view, n_blobs, rng, gen):
    """Fill a 2-D float32 device view with anisotropic Gaussian blobs (centres
    in the inscribed disk, sigma 5 to 40 px) and noise of deviation 0.01."""
    h, w = view.shape
    view.normal_(0.0, 0.01, generator=gen)
    r0 = min(h, w) / 2.0
    for _ in range(n_blobs):
        rr, ph = r0 * math.sqrt(rng.random()), 2 * math.pi * rng.random()
        bx, by = (w - 1) / 2.0 + rr * math.cos(ph), (h - 1) / 2.0 - rr * math.sin(ph)
        s1, s2 = rng.uniform(5.0, 40.0, size=2)
        ang, amp, ext = rng.uniform(0.0, math.pi), rng.uniform(0.2, 1.0), 5.0 * max(s1, s2)
        x0, x1 = max(int(bx - ext), 0), min(int(bx + ext) + 2, w)
        y0, y1 = max(int(by - ext), 0), min(int(by + ext) + 2, h)
        if x0 >= x1 or y0 >= y1:
            continue
        dx = torch.arange(x0, x1, device=view.device, dtype=torch.float32)[None, :] - bx
        dy = torch.arange(y0, y1, device=view.device, dtype=torch.float32)[:, None] - by
        u, v = (dx * math.cos(ang) + dy * math.sin(ang)) / s1, (dy * math.cos(ang) - dx * math.sin(ang)) / s2
        view[y0:y1, x0:x1] += amp * torch.exp(-0.5 * (u * u + v * v))


def _gens(seed, salt):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * (seed % (1 << 40)) + salt)
    return np.random.default_rng([seed % (1 << 63), salt]), gen


def _images(c, seed):
    """The images of a case; a crop is a window of a larger buffer, with rows
    that start on no 16-byte boundary."""
    rng, gen = _gens(seed, 1)
    out = []
    for _ in range(c["batch"]):
        if c.get("crop"):
            base = torch.empty((c["h"] + 2, c["w"] + 6), device="cuda")
            pitch = c["w"] + 5
            view = base.view(-1)[3:3 + pitch * c["h"]].view(c["h"], pitch)[:, :c["w"]]
        else:
            view = torch.empty((c["h"], c["w"]), device="cuda")
        _frame(view, c["blobs"], rng, gen)
        out.append(view)
    return out


def _geometry(c):
    """The disk of a crop sits off its centre; other images use the default."""
    if not c.get("crop"):
        return None
    r = 0.45 * min(c["h"], c["w"])
    return (float(np.float32(c["w"] * 0.48)), float(np.float32(c["h"] * 0.53)), float(np.float32(r)))


def _orders(n_max):
    return [(n, m) for n in range(n_max + 1) for m in range(n % 2, n + 1, 2)]


def _stored_moments(c, seed):
    """Stored moments of `batch` images: complex, falling off with the order as
    those of smooth frames do."""
    rng, _ = _gens(seed, 2)
    nm = np.array(_orders(c["n_max"]))
    z = rng.normal(size=(c["batch"], len(nm), 2)) / (1.0 + nm[:, 0])[None, :, None]
    z[:, nm[:, 1] == 0, 1] = 0.0
    z[:, 0, 0] = 2.0 + rng.random(c["batch"])
    return torch.from_numpy(z.astype(np.float32)).cuda()


def _stored_samples(c, seed):
    """Stored polar samples: a smooth pattern and noise."""
    _, gen = _gens(seed, 3)
    b, nr, nt = c["batch"], c["n_rho"], c["n_theta"]
    f = torch.empty((b, nr, nt), device="cuda")
    f.normal_(0.0, 0.05, generator=gen)
    rho = ((torch.arange(nr, device="cuda") + 0.5) / nr)[None, :, None]
    th = (torch.arange(nt, device="cuda") * (2 * math.pi / nt))[None, None, :]
    k = torch.arange(1, b + 1, device="cuda", dtype=torch.float32)[:, None, None]
    f += 0.5 + 0.3 * rho * torch.cos(th + k) + 0.2 * rho * rho * torch.cos(2 * th - 0.7 * k)
    return f


def _requests(c):
    """(size, n_max, n_rho, n_theta) of an uneven batch."""
    rng = np.random.default_rng(c["spec"])
    reqs = []
    for _ in range(c["batch"]):
        size, n = int(rng.choice([128, 256, 512, 1024])), int(rng.integers(30, 81))
        reqs.append((size, n, size // 2, _theta(n)))
    return reqs


def _request_images(c, seed):
    rng, gen = _gens(seed, 4)
    out = []
    for size, _, _, _ in _requests(c):
        im = torch.empty((size, size), device="cuda")
        _frame(im, 4, rng, gen)
        out.append(im)
    return out


def _pairs(c):
    return [tuple(int(v) for v in p.split(":")) for p in c["pairs"].split(",")]


class _Plan:
    """A plan that is given back with the state that holds it."""

    def __init__(self, c):
        self.h = zm.zm_plan(c["n_max"], c["n_rho"], c["n_theta"], _plan_flags(c))
        zm.zm_plan_reserve(self.h, c["batch"])

    def __del__(self):
        zm.zm_plan_destroy(self.h)


class _Batch:
    def __init__(self, reqs, flags):
        self.h = zm.zm_batch_create(reqs, flags)

    def __del__(self):
        zm.zm_batch_destroy(self.h)


def _plan_flags(c):
    return PREC[c["prec"]] | (zm.ZM_GRID_GAUSS if c["gauss"] else 0)


# ------------------------------------------------------------------ the cases
def prepare(case, seed):
    c = case
    s = {"kind": c["kind"], "flags": zm.ZM_NEUMANN if c["neumann"] else 0, "batch": c["batch"]}
    p = zm.zm_num_moments(c["n_max"])
    if c["kind"] in ("moments", "errors", "recon", "colour", "upload"):
        s["plan"] = _Plan(c)
    polar = (c["batch"], c["n_rho"], c["n_theta"])
    if c["kind"] == "moments":
        s["keep"] = _images(c, seed)
        s["images"] = zm.image_array(s["keep"], [_geometry(c)] * c["batch"])
        s["out"] = torch.empty((c["batch"], p, 2), device="cuda")
    elif c["kind"] == "upload":
        s["host"] = [im.cpu().pin_memory() for im in _images(c, seed)]
        s["dev"] = torch.empty(zm.zm_upload_disk_bytes(s["host"]) // 4 + 4, device="cuda")
        s["out"] = torch.empty((c["batch"], p, 2), device="cuda")
    elif c["kind"] in ("errors", "recon"):
        s["moments"] = _stored_moments(c, seed)
        s["rec"] = torch.empty(polar, device="cuda")
        if c["kind"] == "errors":
            s["fhat"] = _stored_samples(c, seed)
            s["err"] = torch.empty((c["batch"], 4), device="cuda", dtype=torch.float64)
    elif c["kind"] == "colour":
        s["keep"] = _images(c, seed)
        s["moments"] = _stored_moments(c, seed)
        s["canvases"] = torch.empty((c["batch"], c["h"], c["w"]), device="cuda")
        views = [s["canvases"][b] for b in range(c["batch"])]
        s["images"], s["targets"], s["decoded"] = zm.image_array(s["keep"]), zm.canvas_array(views), zm.image_array(views)
        s["polar"] = torch.empty(polar, device="cuda")
        s["minmax"] = torch.empty((c["batch"], 2), device="cuda")
        s["err"] = torch.empty((c["batch"], 4), device="cuda", dtype=torch.float64)
    elif c["kind"] == "cartesian":
        s["keep"] = _images(c, seed)
        s["images"] = zm.image_array(s["keep"])
        s["pairs"] = _pairs(c)
        s["out"] = torch.empty((c["batch"], len(s["pairs"]), 2), device="cuda")
        s["work"] = torch.empty(zm.zm_cartesian_work_bytes(c["batch"], len(s["pairs"])) // 8 + 1, device="cuda",
                                dtype=torch.float64)
    elif c["kind"] == "uneven":
        s["keep"] = _request_images(c, seed)
        # one buffer for the moments of all requests, one after another
        counts = [zm.zm_num_moments(n) for _, n, _, _ in _requests(c)]
        s["out"] = torch.empty((sum(counts), 2), device="cuda")
        s["reqs"] = zm.requests([(im, n, nr, nt, o) for im, (_, n, nr, nt), o in
                                 zip(s["keep"], _requests(c), torch.split(s["out"], counts))])
        s["handle"] = _Batch(s["reqs"], _plan_flags(c))
    return s


def run(state):
    s, flags = state, state["flags"]
    if s["kind"] == "moments":
        zm.zm_moments(s["plan"].h, s["images"], s["out"], flags)
        return s["out"]
    if s["kind"] == "upload":
        boxes = zm.zm_upload_disk(s["host"], s["dev"])
        zm.zm_moments(s["plan"].h, boxes, s["out"], flags)
        return s["out"]
    if s["kind"] == "errors":
        zm.zm_reconstruct_errors(s["plan"].h, s["moments"], s["batch"], s["rec"], s["fhat"], s["err"], flags)
        return {"rec": s["rec"], "err": s["err"]}
    if s["kind"] == "recon":
        zm.zm_reconstruct(s["plan"].h, s["moments"], s["batch"], s["rec"], flags)
        return s["rec"]
    if s["kind"] == "colour":
        zm.zm_disk_minmax(s["plan"].h, s["images"], s["minmax"])
        zm.zm_reconstruct_cartesian(s["plan"].h, s["moments"], s["targets"], s["polar"], flags)
        zm.zm_minmax_normalize(s["plan"].h, s["targets"], s["minmax"])
        zm.zm_errors(s["plan"].h, s["images"], s["decoded"], s["err"])
        return {"minmax": s["minmax"], "polar": s["polar"], "frame": s["canvases"], "err": s["err"]}
    if s["kind"] == "cartesian":
        zm.zm_cartesian_moments(s["images"], s["pairs"], s["out"], s["work"], flags)
        return s["out"]
    zm.zm_batch_run(s["handle"].h, s["reqs"], flags)
    return s["out"]


def _moments_work(h, w, n_max, n_rho, n_theta, batch):
    """Pixels the stencils touch (the disk, or four a sample where those are
    fewer), the radial weights once, the moments; the arithmetic of the bilinear
    samples, the ring FFTs and the radial sums."""
    p = zm.zm_num_moments(n_max)
    px = min(math.pi * (min(h, w) / 2.0) ** 2, 4.0 * n_rho * n_theta)
    rings = n_rho * (7.0 * n_theta + 2.5 * n_theta * math.log2(n_theta))
    return batch * (4.0 * px + 8.0 * p) + 4.0 * p * n_rho, batch * (rings + 4.0 * p * n_rho)


def work(case):
    c = case
    nodes = c["batch"] * c["n_rho"] * c["n_theta"]
    p = zm.zm_num_moments(c["n_max"])
    if c["kind"] == "moments":
        by, fl = _moments_work(c["h"], c["w"], c["n_max"], c["n_rho"], c["n_theta"], c["batch"])
    elif c["kind"] == "upload":
        by, fl = _moments_work(c["h"], c["w"], c["n_max"], c["n_rho"], c["n_theta"], c["batch"])
        by += c["batch"] * 4.0 * math.pi * (min(c["h"], c["w"]) / 2.0) ** 2
    elif c["kind"] in ("errors", "recon", "colour"):
        by = 4.0 * nodes + 4.0 * p * c["n_rho"] + 8.0 * p * c["batch"]
        fl = c["batch"] * (4.0 * p * c["n_rho"] + c["n_rho"] * 2.5 * c["n_theta"] * math.log2(c["n_theta"]))
        if c["kind"] == "errors":
            by, fl = by + 4.0 * nodes, fl + 4.0 * nodes
        if c["kind"] == "colour":
            disk = c["batch"] * math.pi * (min(c["h"], c["w"]) / 2.0) ** 2
            by, fl = by + 4.0 * c["batch"] * c["h"] * c["w"] + 4.0 * disk, fl + 30.0 * disk
    elif c["kind"] == "cartesian":
        disk = c["batch"] * math.pi * (min(c["h"], c["w"]) / 2.0) ** 2
        by, fl = 4.0 * disk, sum(disk * (4.0 + (5.0 * (n - m) / 2 + 10.0) / 8.0) for n, m in _pairs(c))
    else:
        by = fl = 0.0
        for size, n, nr, nt in _requests(c):
            b1, f1 = _moments_work(size, size, n, nr, nt, 1)
            by, fl = by + b1 - 4.0 * zm.zm_num_moments(n) * nr, fl + f1
    return {"bytes": float(by), "flops": float(fl)}


# ------------------------------------------------------------------ 64 bits
def _nodes(n_rho, gauss):
    """Radial nodes and weights (the Jacobian rho included)."""
    if gauss:
        x, w = np.polynomial.legendre.leggauss(n_rho)
        rho = 0.5 * (x + 1.0)
        wr = 0.5 * w * rho
    else:
        rho = (np.arange(n_rho) + 0.5) / n_rho
        wr = rho / n_rho
    return torch.from_numpy(rho).cuda(), torch.from_numpy(wr).cuda()


def _radial(n_max, rho):
    """R_{m+2s, m}(rho) for s = 0, 1, ..: per s a tensor [m][rho] of the orders
    m with m + 2 s <= n_max, from the Jacobi recurrence of P_s^{(0, m)}."""
    m = torch.arange(n_max + 1, device=rho.device, dtype=torch.float64)[:, None]
    x = (2.0 * rho * rho - 1.0)[None, :]
    prev, cur = torch.zeros((n_max + 1, len(rho)), device=rho.device, dtype=torch.float64), rho[None, :] ** m
    for s in range(n_max // 2 + 1):
        live = n_max - 2 * s + 1
        yield s, cur[:live]
        if s == 0:
            nxt = (0.5 * (m + 2.0) * x - 0.5 * m) * cur
        else:
            a, d = 2.0 * s + m, 2.0 * (s + 1.0) * (s + m + 1.0)
            nxt = (((a + 1.0) * (a + 2.0) / d) * x - (a + 1.0) * m * m / (d * a)) * cur - \
                (2.0 * s * (s + m) * (a + 2.0) / (d * a)) * prev
        prev, cur = cur, nxt


def _bilinear(im, x, y):
    h, w = im.shape
    x0, y0 = torch.floor(x), torch.floor(y)
    fx, fy = x - x0, y - y0
    x0, y0 = x0.long(), y0.long()

    def at(xx, yy):
        ok = (xx >= 0) & (xx < w) & (yy >= 0) & (yy < h)
        return torch.where(ok, im[yy.clamp(0, h - 1), xx.clamp(0, w - 1)].double(), 0.0)

    top = (1 - fx) * at(x0, y0) + fx * at(x0 + 1, y0)
    bot = (1 - fx) * at(x0, y0 + 1) + fx * at(x0 + 1, y0 + 1)
    return (1 - fy) * top + fy * bot


def _exact_moments(ims, geo, n_max, n_rho, n_theta, gauss, neumann):
    rho, wr = _nodes(n_rho, gauss)
    th = torch.arange(n_theta, device="cuda", dtype=torch.float64) * (2 * math.pi / n_theta)
    spectra = []
    for im in ims:
        h, w = im.shape
        cx, cy, r = geo or ((w - 1) / 2.0, (h - 1) / 2.0, min(h, w) / 2.0)
        f = _bilinear(im, cx + r * rho[:, None] * torch.cos(th), cy - r * rho[:, None] * torch.sin(th))
        spectra.append(torch.fft.fft(f, dim=1)[:, :n_max + 1].T)
    spectra = torch.stack(spectra)                       # [b][m][rho]
    index = {nm: k for k, nm in enumerate(_orders(n_max))}
    z = torch.zeros((len(ims), len(index)), device="cuda", dtype=torch.complex128)
    for s, rad in _radial(n_max, rho):
        live = rad.shape[0]
        d = torch.einsum("mi,bmi->bm", (rad * wr).to(torch.complex128), spectra[:, :live])
        m = torch.arange(live, device="cuda", dtype=torch.float64)
        d = d * ((m + 2 * s + 1.0) / math.pi * (2 * math.pi / n_theta))
        if neumann:
            d[:, 0] = d[:, 0] / 2.0
        z[:, torch.tensor([index[(k + 2 * s, k)] for k in range(live)], device="cuda")] = d
    return torch.view_as_real(z)


def _exact_polar(c, moments):
    n_max, nt = c["n_max"], c["n_theta"]
    rho, _ = _nodes(c["n_rho"], c["gauss"])
    z = torch.view_as_complex(moments.double().contiguous())
    index = {nm: k for k, nm in enumerate(_orders(n_max))}
    g = torch.zeros((len(z), n_max + 1, c["n_rho"]), device="cuda", dtype=torch.complex128)
    for s, rad in _radial(n_max, rho):
        live = rad.shape[0]
        zs = z[:, torch.tensor([index[(k + 2 * s, k)] for k in range(live)], device="cuda")]
        g[:, :live] += zs[:, :, None] * rad[None]
    if c["neumann"]:
        g[:, 1:] *= 2.0
    full = torch.zeros((len(z), c["n_rho"], nt), device="cuda", dtype=torch.complex128)
    full[:, :, :n_max + 1] = g.transpose(1, 2)
    return (torch.fft.ifft(full, dim=2) * nt).real


def _scores(f, g):
    """(eps_1, eps, f_max, count) over the last dimension."""
    sd, mx, cnt = ((f - g) ** 2).sum(-1), f.amax(-1), float(f.shape[-1])
    return torch.stack([sd / (f ** 2).sum(-1), sd / (mx * mx * cnt), mx, torch.full_like(mx, cnt)], -1)


def _disk(h, w):
    """Pixel offsets from the centre and the disk's mask: sizes in half pixels,
    so that the membership test is exact."""
    x2 = (2 * torch.arange(w, device="cuda") - (w - 1))[None, :]
    y2 = ((h - 1) - 2 * torch.arange(h, device="cuda"))[:, None]
    return x2.double() / 2, y2.double() / 2, x2 * x2 + y2 * y2 <= min(h, w) ** 2


def _exact_colour(c, seed):
    ims, (dx, dy, mask) = _images(c, seed), _disk(c["h"], c["w"])
    mm = torch.stack([torch.stack([im[mask].min(), im[mask].max()]) for im in ims]).double()
    polar = _exact_polar(c, _stored_moments(c, seed))
    rho, _ = _nodes(c["n_rho"], c["gauss"])
    r, nt, nr = min(c["h"], c["w"]) / 2.0, c["n_theta"], c["n_rho"]
    rr = torch.sqrt(dx * dx + dy * dy)[mask] / r
    v = torch.remainder(torch.atan2(dy.expand_as(mask), dx.expand_as(mask))[mask], 2 * math.pi) * (nt / (2 * math.pi))
    i1 = torch.searchsorted(rho, rr, right=True)
    lo, hi = (i1 - 1).clamp(0, nr - 1), i1.clamp(0, nr - 1)
    span = rho[hi] - rho[lo]
    t = torch.where(span > 0, (rr - rho[lo]) / torch.where(span > 0, span, 1.0), 0.0).clamp(0, 1)
    k0 = torch.floor(v).long() % nt
    k1, s = (k0 + 1) % nt, v - torch.floor(v)
    frames, errs = [], []
    for b, im in enumerate(ims):
        pb = polar[b]
        a = pb[lo, k0] * (1 - s) + pb[lo, k1] * s
        o = pb[hi, k0] * (1 - s) + pb[hi, k1] * s
        val = a * (1 - t) + o * t
        g0, g1 = val.min(), val.max()
        val = (val - g0) * ((mm[b, 1] - mm[b, 0]) / (g1 - g0)) + mm[b, 0]
        fr = torch.zeros((c["h"], c["w"]), device="cuda", dtype=torch.float64)
        fr[mask] = val
        frames.append(fr)
        errs.append(_scores(im[mask].double(), val))
    return {"minmax": mm, "polar": polar, "frame": torch.stack(frames), "err": torch.stack(errs)}


def _exact_cartesian(c, seed):
    dx, dy, mask = _disk(c["h"], c["w"])
    r = min(c["h"], c["w"]) / 2.0
    x, y = (dx.expand_as(mask)[mask] / r), (dy.expand_as(mask)[mask] / r)
    rho2, th = x * x + y * y, torch.atan2(y, x)
    out = torch.zeros((c["batch"], len(_pairs(c)), 2), device="cuda", dtype=torch.float64)
    ims = [im[mask].double() for im in _images(c, seed)]
    for k, (n, m) in enumerate(_pairs(c)):
        prev, cur, xx = torch.zeros_like(rho2), rho2 ** (m / 2.0), 2.0 * rho2 - 1.0
        for s in range((n - m) // 2):
            if s == 0:
                nxt = (0.5 * (m + 2.0) * xx - 0.5 * m) * cur
            else:
                a, d = 2.0 * s + m, 2.0 * (s + 1.0) * (s + m + 1.0)
                nxt = (((a + 1.0) * (a + 2.0) / d) * xx - (a + 1.0) * m * m / (d * a)) * cur - \
                    (2.0 * s * (s + m) * (a + 2.0) / (d * a)) * prev
            prev, cur = cur, nxt
        scale = (n + 1) / (math.pi * r * r) / (2.0 if c["neumann"] and m == 0 else 1.0)
        re, im_ = cur * torch.cos(m * th), cur * torch.sin(m * th)
        for b, f in enumerate(ims):
            out[b, k, 0], out[b, k, 1] = scale * (f * re).sum(), -scale * (f * im_).sum()
    return out


def exact(case, seed):
    c = case
    if c["kind"] in ("moments", "upload"):
        return _exact_moments(_images(c, seed), _geometry(c), c["n_max"], c["n_rho"], c["n_theta"], c["gauss"],
                              c["neumann"])
    if c["kind"] == "uneven":
        return torch.cat([_exact_moments([im], None, n, nr, nt, c["gauss"], c["neumann"])[0]
                          for im, (_, n, nr, nt) in zip(_request_images(c, seed), _requests(c))])
    if c["kind"] == "recon":
        return _exact_polar(c, _stored_moments(c, seed))
    if c["kind"] == "errors":
        rec, f = _exact_polar(c, _stored_moments(c, seed)), _stored_samples(c, seed).double()
        return {"rec": rec, "err": _scores(f.reshape(len(f), -1), rec.reshape(len(f), -1))}
    if c["kind"] == "colour":
        return _exact_colour(c, seed)
    return _exact_cartesian(c, seed)
