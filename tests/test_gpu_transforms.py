"""The row and column transforms at every length the launches choose between
(images of 32 to 2048 pixels, so transforms of 64 to 8192 points with the
PSF's grid; one to many rows or columns per CTA; narrow and nearly full uv
windows), through degrid, grid and PSF of a few hundred samples against the
direct DFT.

Tolerances: the exponential-of-semicircle kernel's own error is below 1e-7 at
these w ranges (dw |n - 1| < 0.11); FP32 adds the rounding of two passes and
of the gridding, a few times 1e-7, so 1e-5 leaves an order of magnitude and
any misplaced or dropped value is far above it; FP64 1e-6."""
import numpy as np
import pytest

from gpu_util import cplx_dtype, need_gpu, real_dtype, rel_l2, sparse_model, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CELL = np.pi / 180 / 3600


def _phase(u, v, w, b, a, n, wterm):
    l, m = (a - n // 2) * CELL, (b - n // 2) * CELL
    r2 = l * l + m * m
    nm1 = -r2 / (1.0 + np.sqrt(1.0 - r2))
    ph = np.outer(u, l) + np.outer(v, m)
    return (ph + np.outer(w, nm1) if wterm else ph), (1.0 + nm1 if wterm else np.ones_like(l))


@pytest.mark.parametrize("reach", [0.07, 0.46])
@pytest.mark.parametrize("planes", [0, 9])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [32, 64, 128, 256, 512, 1024, 2048])
def test_operator_against_direct_dft(n, prec, planes, reach):
    need_gpu()
    from paper_2507_22128_gb300 import rix
    rng = np.random.default_rng(n + 7 * planes + prec)
    ns, tol = 301, (1e-5 if prec == rix.FP32 else 1e-6)
    wave = 299792458.0 / 1.4e9
    lim = min(reach, 0.5 - 5.0 / (2 * n)) / CELL
    uvw = np.stack([rng.uniform(-lim, lim, ns), rng.uniform(-lim, lim, ns), rng.uniform(-2000, 2000, ns)], 1) * wave
    u, v, w = (uvw * (1.4e9 / 299792458.0)).T
    vis = rng.normal(size=ns) + 1j * rng.normal(size=ns)
    ctx = rix.create(0)
    job = rix.job_create(ctx, n, CELL, planes, [1.4e9], prec, 1, ns)
    try:
        rix.set_uv_partition(job, to_dev(uvw, torch.float64))
        assert rix.job_get_stats(job)["n_outside"] == 0
        x = sparse_model(n, 12, 3)
        b, a = np.nonzero(x)
        ph, nn = _phase(u, v, w, b, a, n, planes > 0)
        want = np.exp(-2j * np.pi * ph) @ (x[b, a] / nn)
        out = torch.zeros(ns, dtype=cplx_dtype(prec), device="cuda")
        rix.degrid(job, 0, to_dev(x, real_dtype(prec)), out)
        assert rel_l2(out.cpu().numpy(), want) < tol
        # the PSF's transforms (side 4N) on coplanar jobs: over the 2N field w-planes spaced for
        # the N field have no bound of this kind (dw |n - 1| reaches 0.4 at 2048)
        checks = [(n, vis, lambda o: rix.grid(job, 0, to_dev(vis, cplx_dtype(prec)), o))]
        if planes == 0:
            checks.append((2 * n, np.ones(ns), lambda o: rix.psf(job, 0, o)))
        for side, y, call in checks:
            img = torch.empty((side, side), dtype=real_dtype(prec), device="cuda")
            call(img)
            b, a = rng.integers(0, side, 200), rng.integers(0, side, 200)
            b[:4], a[:4] = [0, 0, side - 1, side // 2], [0, side - 1, 1, side // 2]
            ph, nn = _phase(u, v, w, b, a, side, planes > 0)
            want = (y @ np.exp(2j * np.pi * ph)).real / nn / ns
            assert np.max(np.abs(img.cpu().numpy()[b, a] - want)) < tol * np.linalg.norm(y) / np.sqrt(ns) * \
                max(1.0, np.max(np.abs(want)))
    finally:
        rix.job_destroy(job)
        rix.destroy(ctx)
