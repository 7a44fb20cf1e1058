"""Jobs of different image sizes driven from two host threads at once, as the
library allows: every call of either thread succeeds and every result is the
one the job gives alone."""
import threading

import numpy as np
import pytest

from gpu_util import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_msclean_of_two_sizes_from_two_threads():
    """ms-CLEAN at 512^2 and 2048^2 shares one kernel instance (32 x 32 tiles, one
    scale) whose shared memory differs with the size.  FP64: the same components
    each time, amplitudes within 1e-9 of the largest."""
    need_gpu()
    from paper_2507_22128_gb300 import pipeline, rix, synth
    m = pipeline.Method("msclean", (0.0,), 0.1, 4, 0.0)
    ctx = rix.create(0)
    recs, errors = [], []
    try:
        obs = [synth.medium(seed=5, n_times=3, n=n, n_ant=10, n_chan=1, n_wplanes=0) for n in (512, 2048)]
        recs = [pipeline.observation_job(ctx, o, 1, rix.FP64) for o in obs]

        def cycles(k, start, out):
            try:
                rec, stream = recs[k], torch.cuda.Stream()
                rec.set_data(obs[k].uvw, obs[k].vis, obs[k].weight)
                torch.cuda.synchronize()
                start.wait()
                for _ in range(60):
                    rec.major(0, stream=stream)
                    rec.minor(0, m, stream=stream)
                stream.synchronize()
                rix.job_sync(rec.job)
                out[k] = rix.get_components(rec.job, 0)
            except Exception as e:   # reported by the test's own thread
                errors.append(f"{obs[k].n}^2: {e}")
                start.abort()

        alone, together = {}, {}
        for k in (0, 1):
            cycles(k, threading.Barrier(1), alone)
        both = threading.Barrier(2)
        threads = [threading.Thread(target=cycles, args=(k, both, together)) for k in (0, 1)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not errors, errors
        for k in (0, 1):
            (s0, p0, a0), (s1, p1, a1) = alone[k], together[k]
            assert np.array_equal(s0, s1) and np.array_equal(p0, p1)
            assert np.abs(a0 - a1).max() <= 1e-9 * np.abs(a0).max()
    finally:
        for r in recs:
            r.close()
        rix.destroy(ctx)
