"""FISTA loops around the 256 iterations whose momentum travels in the launch
arguments: the cluster, the single loop on the grid and the concatenated dictionary
go on from its last value on the device, a batch takes a table instead.  FP64
against the oracle's minor cycle within 1e-9, the bound of the FISTA loops."""
import pytest

from gpu_util import need_gpu, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nparts,iters,dictionary", [
    (32, 1, 255, "db4"), (32, 1, 256, "db4"), (32, 1, 257, "db4"), (64, 2, 260, "db4"), (32, 1, 259, "db1-8"),
    (256, 1, 256, "db4"), (256, 1, 260, "db4"), (256, 2, 256, "db4"), (256, 2, 260, "db4")])
def test_long_minor_cycle_matches_the_oracle(n, nparts, iters, dictionary):
    need_gpu()
    from oracle import framework
    from paper_2507_22128_gb300 import pipeline, rix, synth
    obs = synth.medium(seed=43, n_times=5, n=n, n_ant=16, n_chan=1, n_wplanes=0)
    loop = framework.Loop(framework.setup(obs.uvw, obs.freq, obs.weight, obs.n, obs.cell_rad, 0, nparts), obs.vis,
                          obs.weight)
    ctx = rix.create(0)
    try:
        with pipeline.observation_job(ctx, obs, nparts, rix.FP64) as rec:
            for p in range(nparts):
                loop.major(p)
                rec.major(p)
            for p in range(nparts):
                loop.minor_fista(p, 1, lam_rel=1e-3, n_iter=iters, levels=2,
                                 dictionary="db4" if dictionary == "db4" else "sara")
            rec.minor_all(pipeline.Method("fista", lam_rel=1e-3, iters=iters, levels=2, dictionary=dictionary),
                          torch.cuda.current_stream())
            loop.exchange()
            assert rel_l2(rec.combine().cpu().numpy(), loop.combine()) < 1e-9
    finally:
        rix.destroy(ctx)
