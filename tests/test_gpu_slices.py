"""Work items cut into slices (k_tiles, k_tiles_ws) or chunks (k_tiles_fp): sample
counts on both sides of the slice and item sizes, all in one or two uv tiles, degrid and grid
of every precision and w-mode that uses them, against the direct DFT.

Tolerances (relative L2): FP32 1e-5 (kernel error 1e-7, a few roundings per
tap), FP64 1e-6 (kernel error); a slice left out, repeated or cut short is at
least 1 / count, 2e-4 here."""
import numpy as np
import pytest

from gpu_util import cplx_dtype, need_gpu, real_dtype, rel_l2, sparse_model, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CELL = np.pi / 180 / 3600


@pytest.mark.parametrize("prec,planes,tile", [(0, 0, 16), (0, 0, 32), (0, 9, 16), (1, 0, 16), (1, 9, 16)])
@pytest.mark.parametrize("ns", [1, 63, 64, 65, 257, 2047, 2048, 2049, 4999])
def test_crowded_tile(ns, prec, planes, tile):
    need_gpu()
    from paper_2507_22128_gb300 import rix
    n, freq, tol = 64, 1.4e9, (1e-5 if prec == rix.FP32 else 1e-6)
    rng = np.random.default_rng(ns)
    uvl = rng.uniform(-3, 3, (ns, 2)) / (2 * n * CELL)       # within three cells of the centre
    wl = rng.uniform(-500, 500, ns)
    uvw = np.column_stack([uvl, wl]) * (299792458.0 / freq)
    off = (np.arange(n) - n // 2) * CELL
    l, m = off[None, :], off[:, None]
    r2 = (l * l + m * m).ravel()
    nm1 = -r2 / (1 + np.sqrt(1 - r2)) if planes else 0 * r2
    ph = np.outer(uvl[:, 0], np.broadcast_to(l, (n, n)).ravel()) + \
        np.outer(uvl[:, 1], np.broadcast_to(m, (n, n)).ravel()) + np.outer(wl, nm1)
    e = np.exp(-2j * np.pi * ph)
    x = sparse_model(n, 9, 1)
    vis = rng.normal(size=ns) + 1j * rng.normal(size=ns)
    wt = rng.uniform(0.5, 1.5, ns).astype(np.float32)
    ctx = rix.create(0)
    job = rix.job_create(ctx, n, CELL, planes, [freq], prec, 1, ns, tile)
    try:
        rix.set_uv_partition(job, to_dev(uvw, torch.float64), to_dev(wt, torch.float32))
        out = torch.zeros(ns, dtype=cplx_dtype(prec), device="cuda")
        rix.degrid(job, 0, to_dev(x, real_dtype(prec)), out)
        assert rel_l2(out.cpu().numpy(), e @ (x.ravel() / (1 + nm1))) < tol
        img = torch.empty((n, n), dtype=real_dtype(prec), device="cuda")
        rix.grid(job, 0, to_dev(vis, cplx_dtype(prec)), img)
        want = ((wt * vis) @ e.conj()).real / (1 + nm1) / wt.astype(np.float64).sum()
        assert rel_l2(img.cpu().numpy().ravel(), want) < tol
    finally:
        rix.job_destroy(job)
        rix.destroy(ctx)
