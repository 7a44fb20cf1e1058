"""Coplanar gridding of samples spread thinly over 16,000 uv tiles with one crowded
tile among them: the CTAs skip the empty slices of most work items, several hundred
candidates each.  Degrid of a few points and the dirty image at sampled pixels
against the direct transform in FP64, relative L2 1e-5 in FP32 (kernel error 1e-7, a
few roundings per tap) and 1e-6 in FP64 (kernel error); a slice left out is at least
1 / 205,000 of the sum, and some 1,000 of them with a wrong range far above both."""
import numpy as np
import pytest

from gpu_util import cplx_dtype, need_gpu, real_dtype, rel_l2, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CELL = np.pi / 180 / 3600


@pytest.mark.parametrize("prec", [0, 1])
def test_thin_and_crowded(prec):
    need_gpu()
    from paper_2507_22128_gb300 import rix
    n, freq, tol = 1024, 1.4e9, (1e-5 if prec == rix.FP32 else 1e-6)
    rng = np.random.default_rng(3)
    grid = np.concatenate([rng.uniform(-1010, 1010, (200000, 2)), rng.uniform(40.0, 52.0, (5000, 2))])
    uvl = grid[rng.permutation(len(grid))] / (2 * n * CELL)
    ns = len(uvl)
    uvw = np.column_stack([uvl, np.zeros(ns)]) * (299792458.0 / freq)
    wt = rng.uniform(0.5, 1.5, ns).astype(np.float32)
    vis = to_dev(rng.normal(size=ns) + 1j * rng.normal(size=ns), cplx_dtype(prec))
    pts = rng.integers(100, 900, (7, 2))
    x = torch.zeros((n, n), dtype=real_dtype(prec), device="cuda")
    x[pts[:, 0], pts[:, 1]] = 1.0
    uv = to_dev(uvl, torch.float64)

    def phase(pix):
        lm = to_dev((pix[:, ::-1] - n // 2) * CELL, torch.float64)
        return torch.exp(-2j * np.pi * (uv @ lm.T))

    look = rng.integers(0, n, (200, 2))
    y = to_dev(wt, torch.float64) * vis.to(torch.complex128)
    want = (phase(look).conj().T @ y).real / float(wt.astype(np.float64).sum())
    ctx = rix.create(0)
    job = rix.job_create(ctx, n, CELL, 0, [freq], prec, 1, ns, 16)
    try:
        rix.set_uv_partition(job, to_dev(uvw, torch.float64), to_dev(wt, torch.float32))
        out = torch.zeros(ns, dtype=cplx_dtype(prec), device="cuda")
        rix.degrid(job, 0, x, out)
        assert rel_l2(out.cpu().numpy(), phase(np.unique(pts, axis=0)).sum(1).cpu().numpy()) < tol
        img = torch.empty((n, n), dtype=real_dtype(prec), device="cuda")
        rix.grid(job, 0, vis, img)
        assert rel_l2(img[look[:, 0], look[:, 1]].cpu().numpy(), want.cpu().numpy()) < tol
    finally:
        rix.job_destroy(job)
        rix.destroy(ctx)
