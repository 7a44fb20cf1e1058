"""FISTA loops at the image sizes their launches choose between (a cluster per
loop up to 128^2, the whole grid from 256^2; one loop and two; both
dictionaries; one to all wavelet levels) against the oracle's minor cycle: FP64
within 1e-9, FP32 within 1e-4, the bounds of the FISTA loops."""
import numpy as np
import pytest

from gpu_util import need_gpu, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dictionary", ["db4", "db1-8"])
@pytest.mark.parametrize("prec", [1, 0])
@pytest.mark.parametrize("n,nparts,levels", [(32, 1, 2), (32, 2, 1), (64, 3, 3), (128, 2, 4), (128, 1, 1),
                                             (256, 2, 5), (256, 1, 3)])
def test_minor_cycles_match_the_oracle(n, nparts, levels, prec, dictionary):
    need_gpu()
    from oracle import framework
    from paper_2507_22128_gb300 import pipeline, rix, synth
    obs = synth.medium(seed=41, n_times=5, n=n, n_ant=16, n_chan=1, n_wplanes=0)
    st = framework.setup(obs.uvw, obs.freq, obs.weight, obs.n, obs.cell_rad, 0, nparts)
    loop = framework.Loop(st, obs.vis, obs.weight)
    ctx = rix.create(0)
    try:
        with pipeline.observation_job(ctx, obs, nparts, prec) as rec:
            m = pipeline.Method("fista", lam_rel=1e-3, iters=7, levels=levels, dictionary=dictionary)
            for c in (1, 2):
                for p in range(nparts):
                    loop.major(p)
                    rec.major(p)
                for p in range(nparts):
                    loop.minor_fista(p, c, lam_rel=1e-3, n_iter=7, levels=levels,
                                     dictionary="db4" if dictionary == "db4" else "sara")
                rec.minor_all(m, torch.cuda.current_stream())
                loop.exchange()
            assert rel_l2(rec.combine().cpu().numpy(), loop.combine()) < (1e-9 if prec == 1 else 1e-4)
    finally:
        rix.destroy(ctx)
