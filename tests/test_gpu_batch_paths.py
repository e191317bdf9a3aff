"""Uneven batches under the environment's resampling switches, and with a tune
cache written before its entries had a version."""

import json

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2304_14492_gb300 import native as zm, synth  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
GROUPS = [(128, 40, 64, 128), (256, 60, 128, 256)]           # size, n_max, n_rho, n_theta


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2304_14492_gb300.build import build
    build()
    zm.lib()


def requests():
    items = []
    for j, (size, n_max, n_rho, n_theta) in enumerate(GROUPS * 3):
        t = torch.from_numpy(synth.blob_image(size, size, 5, workload=42, index=j)).to(DEV)
        items.append((t, n_max, n_rho, n_theta, torch.full((zm.zm_num_moments(n_max), 2), float("nan"), device=DEV)))
    return items


def run(items, prec):
    """Outputs of a batch, the library's launches in one capture of it, and the
    outputs of zm_moments on plans made under the same environment."""
    batch = zm.zm_batch_create(items, prec)
    try:
        zm.zm_batch_run(batch, items)
        torch.cuda.synchronize()
        outs = [it[4].clone() for it in items]
        again = [it[:4] + (torch.empty_like(it[4]),) for it in items]
        before = zm.zm_launch_count()
        zm.zm_batch_run(batch, again)                        # new pointers: captured again
        launches = zm.zm_launch_count() - before
        torch.cuda.synchronize()
    finally:
        zm.zm_batch_destroy(batch)
    alone = []
    for t, n_max, n_rho, n_theta, out in items:
        plan = zm.zm_plan(n_max, n_rho, n_theta, prec)
        try:
            o = torch.empty((1,) + tuple(out.shape), device=DEV)
            zm.zm_moments(plan, [t], o)
            torch.cuda.synchronize()
        finally:
            zm.zm_plan_destroy(plan)
        alone.append(o[0])
    return outs, launches, alone


@pytest.mark.parametrize("fused", ["0", "1"])
def test_fused_switch_reaches_batches(fused, tmp_path, monkeypatch):
    cache = tmp_path / "tune.json"
    monkeypatch.setenv("ZM_TUNE_CACHE", str(cache))
    plain, n_plain, _ = run(requests(), zm.ZM_PREC_BF16X3)
    assert [v["gather"] for v in json.load(open(cache)).values()] == [1, 1]
    monkeypatch.setenv("ZM_FUSED", fused)
    outs, n, _ = run(requests(), zm.ZM_PREC_BF16X3)
    assert all(torch.equal(a, b) for a, b in zip(plain, outs))
    # two launches a group (gathered or staged, then the projection), three with
    # the tiles, and the copies
    assert n_plain == 2 * len(GROUPS) + 1 and n == (2 if fused == "1" else 3) * len(GROUPS) + 1
    new = [v["gather"] for k, v in json.load(open(cache)).items() if "|fused=%d|" % (1 if fused == "1" else -1) in k]
    assert new == [0, 0]


def test_tensor_core_transform_reaches_batches(monkeypatch):
    plain, _, _ = run(requests(), zm.ZM_PREC_BF16X3)
    monkeypatch.setenv("ZM_RING_DFT", "1")
    outs, _, alone = run(requests(), zm.ZM_PREC_BF16X3)
    for a, b, c in zip(plain, outs, alone):
        assert torch.equal(b, c)                             # the transform that zm_moments takes
        assert not torch.equal(a, b)                         # (whose roundings are not the FFT's)
        assert float((a - b).abs().max()) <= 2e-5 * float(a.abs().max())


def test_entries_without_a_version_are_kept_and_not_read(tmp_path, monkeypatch):
    cache = tmp_path / "tune.json"
    monkeypatch.setenv("ZM_TUNE_CACHE", str(cache))
    cap = torch.cuda.get_device_capability()
    old = {"sm%d%d|nrho=%d|ntheta=%d|nmax=%d|batch=4|prec=%d|grid=0|img=%dx%d"
           % (cap[0], cap[1], r, t, n, p, s, s): {"gather": 0, "rings": 8, "split": 8, "us": 1.0}
           for s, n, r, t in GROUPS for p in (0, 1)}
    with open(cache, "w") as f:
        f.write("{\n" + ",\n".join('  "%s": {"gather": 0, "rings": 8, "split": 8, "us": 1.000}' % k for k in old) + "\n}\n")
    run(requests(), zm.ZM_PREC_BF16X3)
    entries = json.load(open(cache))
    new = [v for k, v in entries.items() if k not in old]
    assert set(old) <= set(entries) and len(new) == len(GROUPS) and all(v["gather"] == 1 for v in new)
