"""FP32 coplanar gridding of one crowded uv tile with entry counts on both sides of
where the slices' length changes (slice_rule.cuh: 64, 128 and 2048 entries, and
whole items), degrid and grid, against a direct transform in FP64.

Tolerance (relative L2) 1e-5, that of the smaller counts: kernel error 1e-7 and a few
roundings per tap; a slice left out, repeated or cut short is at least
64 / 93,000 = 7e-4."""
import numpy as np
import pytest

from gpu_util import need_gpu, rel_l2, sparse_model, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CELL = np.pi / 180 / 3600


@pytest.mark.parametrize("tile", [16, 32])
@pytest.mark.parametrize("ns", [16639, 16641, 23999, 92681, 92683])
def test_crowded_tile(ns, tile):
    need_gpu()
    from paper_2507_22128_gb300 import rix
    n, freq = 64, 1.4e9
    rng = np.random.default_rng(ns)
    uvl = rng.uniform(-3, 3, (ns, 2)) / (2 * n * CELL)       # within three cells of the centre
    uvw = np.column_stack([uvl, np.zeros(ns)]) * (299792458.0 / freq)
    wt = to_dev(rng.uniform(0.5, 1.5, ns), torch.float32)
    vis = to_dev(rng.normal(size=ns) + 1j * rng.normal(size=ns), torch.complex64)
    x = to_dev(sparse_model(n, 9, 1), torch.float32)
    off = to_dev((np.arange(n) - n // 2) * CELL, torch.float64)
    uv = to_dev(uvl, torch.float64)
    # e^(-2 pi i u l) per sample and pixel column, e^(-2 pi i v m) per sample and row
    eu, ev = (torch.exp(-2j * np.pi * uv[:, k:k + 1] * off) for k in (0, 1))
    model = torch.einsum("sm,ml,sl->s", ev, x.to(torch.complex128), eu)
    dirty = ((wt.double() * vis.to(torch.complex128))[:, None] * ev.conj()).T @ eu.conj()
    ctx = rix.create(0)
    job = rix.job_create(ctx, n, CELL, 0, [freq], rix.FP32, 1, ns, tile)
    try:
        rix.set_uv_partition(job, to_dev(uvw, torch.float64), wt)
        out = torch.zeros(ns, dtype=torch.complex64, device="cuda")
        rix.degrid(job, 0, x, out)
        assert rel_l2(out.cpu().numpy(), model.cpu().numpy()) < 1e-5
        img = torch.empty((n, n), dtype=torch.float32, device="cuda")
        rix.grid(job, 0, vis, img)
        assert rel_l2(img.cpu().numpy(), (dirty.real / wt.double().sum()).cpu().numpy()) < 1e-5
    finally:
        rix.job_destroy(job)
        rix.destroy(ctx)
