"""The calls a user of this library spends device time in, with their inputs.

Five operations, each through the public binding (`rix`) or the host driver
(`pipeline`):

* ``predict``  rix.degrid of every partition: model image -> visibilities;
* ``image``    rix.grid of every partition: visibilities -> dirty images;
* ``major``    the fused major cycle (degrid, residual, grid) of every
               partition of one or more jobs, replayed from the CUDA graph of
               pipeline.BatchedMajor;
* ``setup``    what every job pays once: coordinates, uv partition, tile sort
               and the partitions' PSFs;
* ``job``      a whole reconstruction (set-up, cycles, combine) with FISTA or
               multi-scale CLEAN minor cycles.

Observations are seeded: antennas on a jittered log spiral (or in a disk),
Earth-rotation uvw tracks, a sky of point sources and circular Gaussians,
analytic visibilities with noise, and weights that vary by sample with a few
flagged (zero) ones.  Row counts are cut to the requested number of samples,
so they are not multiples of anything.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_22128_gb300 import pipeline, rix

C_LIGHT = 299792458.0
ARCSEC = math.pi / (180.0 * 3600.0)
DEV = "cuda"

_BASE = {"op": "", "n": 128, "planes": 0, "nvis": 0, "nchan": 1, "ants": 32, "radius_m": 1000.0, "cell_as": 2.0,
         "hours": 4.0, "parts": 2, "fp64": False, "weights": True, "uniform": False, "spectral": False, "pts": 24,
         "gauss": 0, "batch": "", "method": "", "cycles": 0, "iters": 0, "levels": 4, "scales": "", "concat": False,
         "sched_a": 0.0, "sched_b": 1.0}


def _case(**kw):
    c = dict(_BASE)
    c.update(kw)
    return c


def _spiral(**kw):
    """The 64-antenna, 5 km log-spiral array at 1" cells of the 1024^2 observations."""
    return _case(**{**dict(n=1024, planes=16, nchan=4, ants=64, radius_m=5000.0, cell_as=1.0, pts=40), **kw})


def listed():
    return [
        # the smallest calls: one snapshot-sized observation of a compact array, coplanar,
        # interactive prediction and imaging; launches and latency count
        _case(name="predict_small", op="predict", nvis=19840, pts=10),
        _case(name="image_small", op="image", nvis=19841, pts=10, weights=False),
        # model visibilities of a full observation, for calibration or subtraction
        _spiral(name="predict_medium", op="predict", nvis=8064000),
        # dirty images of a full observation under uniform weighting
        _spiral(name="image_medium", op="image", nvis=7999996, uniform=True),
        # major cycles of a batch of channel chunks of several image sizes at once
        _spiral(name="major_chunks", op="major", n=2048,
                batch="256x601132,512x3203476,1024x1100020,2048x2101104,1024x4000004"),
        # the largest images: 4096^2 at 0.5", 32 w-planes, 8 channels, a 10 km array of 128 antennas
        _case(name="major_large", op="major", n=4096, planes=32, nvis=16000000, nchan=8, ants=128, radius_m=10000.0,
              cell_as=0.5, pts=40, batch="4096x16000000"),
        # what every full-size job pays before its first major cycle
        _spiral(name="setup_medium", op="setup", nvis=8064000),
        # whole jobs: the small observation, many of which a server runs
        _case(name="job_small", op="job", nvis=19840, pts=10, gauss=2, method="fista", cycles=5, iters=50, levels=4),
        # the full observation with FISTA on a Db4 basis, the library's main workload
        _spiral(name="job_medium", op="job", nvis=8064000, gauss=8, method="fista", cycles=5, iters=50),
        # multi-scale CLEAN of a wide field with the scales of the large observations
        _spiral(name="job_clean_wide", op="job", n=2048, nvis=1500000, gauss=4, pts=12, method="msclean", cycles=1,
                iters=300, scales="0,4,16,32"),
        # the method as published: concatenated db1 .. db8 dictionary, lambda schedule, uniform weighting
        _spiral(name="job_concat", op="job", n=512, nvis=1000000, gauss=6, method="fista", cycles=2, iters=50,
                concat=True, sched_a=0.002, sched_b=0.7, uniform=True),
        # double precision: three rings, w-stacked, CLEAN to a fixed number of components
        _spiral(name="job_fp64", op="job", n=512, planes=12, nvis=400003, nchan=1, fp64=True, parts=3, gauss=4,
                pts=12, method="msclean", cycles=2, iters=200, scales="0,4,16"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choice(["predict", "image", "major", "setup", "job"])
    fp64 = op in ("predict", "image", "setup") and rng.random() < 0.25
    coplanar = op != "major" and rng.random() < 0.25
    n = rng.choice([64, 128, 256, 512] if (fp64 or coplanar) else [128, 256, 512, 1024, 2048])
    nvis = int(_log(rng, 5e3, 4e5 if fp64 else 6e6)) | 1
    nchan = rng.choice([1, 2, 3, 4, 8])
    kw = dict(op=op, n=n, planes=0 if coplanar else rng.randint(9, 24), nvis=nvis, nchan=nchan, fp64=fp64,
              parts=rng.randint(1, 4), uniform=rng.random() < 0.3, weights=rng.random() < 0.7,
              ants=rng.choice([27, 32, 45, 64]), radius_m=_log(rng, 1500.0, 6000.0), pts=rng.randint(8, 40))
    if op == "major":
        sizes = [(n, nvis)] + [(rng.choice([128, 256, 512, 1024]), int(_log(rng, 5e4, 2e6)) | 1)
                               for _ in range(rng.randint(0, 3))]
        kw["batch"] = ",".join(f"{a}x{b}" for a, b in sizes)
    if op == "job":
        n = min(n, 1024)
        kw.update(n=n, nvis=min(nvis, 2000001), gauss=rng.randint(0, 6), cycles=rng.randint(1, 3), pts=12,
                  spectral=rng.random() < 0.25)
        if rng.random() < 0.5:
            concat = rng.random() < 0.3
            kw.update(n=min(n, 256) if concat else n, method="fista", iters=rng.randint(10, 50),
                      levels=rng.randint(2, 4), concat=concat)
        else:
            # double precision where its cost allows: greedy choices then do not hang on rounding
            kw.update(method="msclean", fp64=n <= 512, nvis=min(kw["nvis"], 300001), iters=rng.randint(50, 200),
                      scales=rng.choice(["0", "0,3,9", "0,4,16"]), cycles=rng.randint(1, 2))
        kw["levels"] = min(kw.get("levels", 4), int(math.log2(kw["n"])) - 3)
    return _spiral(**kw)


# ------------------------------------------------------------------ inputs ----
def _rng(seed, salt=0):
    return np.random.Generator(np.random.PCG64(np.random.SeedSequence([int(seed), salt])))


def _observation(case, seed, nvis):
    """uvw (metres), frequencies, sky and weights of `nvis` samples (rounded down to whole rows)."""
    g = _rng(seed)
    na = case["ants"]
    if case["planes"]:
        arm = np.arange(na) % 3
        r = np.geomspace(0.01 * case["radius_m"], case["radius_m"], na) * g.uniform(0.95, 1.0, na)
        th = 2.0 * np.pi * arm / 3.0 + 1.2 * np.log(r / r.min()) + g.normal(0.0, 0.02, na)
    else:
        r = case["radius_m"] * np.sqrt(g.random(na))
        th = 2.0 * np.pi * g.random(na)
    e, nn = r * np.cos(th), r * np.sin(th)
    i, j = np.triu_indices(na, k=1)
    nchan = case["nchan"]
    nrow = max(nvis // nchan, 1)
    n_times = -(-nrow // i.size)
    ha = np.linspace(-0.5 * case["hours"], 0.5 * case["hours"], max(n_times, 2))[:n_times] * (math.pi / 12.0)
    lat = dec = -math.pi / 6.0
    t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=DEV)
    x = t(-math.sin(lat) * (nn[j] - nn[i]))
    y = t(e[j] - e[i])
    z = t(math.cos(lat) * (nn[j] - nn[i]))
    sh, ch = t(np.sin(ha))[:, None], t(np.cos(ha))[:, None]
    sd, cd = math.sin(dec), math.cos(dec)
    uvw = torch.stack([sh * x + ch * y, -sd * ch * x + sd * sh * y + cd * z, cd * ch * x - cd * sh * y + sd * z], -1)
    uvw = uvw.reshape(-1, 3)[:nrow].contiguous()
    freq = np.linspace(1.3e9, 1.5e9, nchan) if nchan > 1 else np.array([1.4e9])
    weight = None
    if case["weights"]:
        gen = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 11)
        weight = 0.5 + torch.rand((nrow, nchan), generator=gen, device=DEV, dtype=torch.float32)
        weight *= torch.rand((nrow, nchan), generator=gen, device=DEV) > 0.02
    return uvw, freq, weight


def _sky(case, seed, n):
    """Pixel offsets and float32 fluxes of the points; the Gaussians' offsets, fluxes and sigmas (pixels)."""
    g = _rng(seed, 1)
    half = int(0.4 * n)
    k = case["pts"]
    pix = g.choice((2 * half) ** 2, size=k, replace=False)
    px, py = pix % (2 * half) - half, pix // (2 * half) - half
    flux = ((1e-2 ** -0.6 + g.random(k) * (1.0 - 1e-2 ** -0.6)) ** (1.0 / -0.6)).astype(np.float32)
    m = case["gauss"]
    return (px, py, flux), (g.integers(-half, half, m), g.integers(-half, half, m), g.uniform(0.1, 1.0, m),
                            g.uniform(1.3, 3.4, m))


def _lambdas(uvw, freq):
    return torch.as_tensor(freq / C_LIGHT, dtype=torch.float64, device=DEV)


def _vis(case, uvw, freq, pts, gauss, cell):
    """Visibilities of the sky in 64 bits, [nrow][nchan] complex128."""
    wterm = case["planes"] > 0
    inv = _lambdas(uvw, freq)
    out = torch.zeros((uvw.shape[0], inv.numel()), dtype=torch.complex128, device=DEV)
    for (dx, dy, fl), sig in ((pts, None), (gauss[:3], gauss[3])):
        if len(fl) == 0:
            continue
        l, m = np.asarray(dx) * cell, np.asarray(dy) * cell
        nn = np.sqrt(1.0 - l * l - m * m)
        amp = torch.as_tensor(np.asarray(fl, np.float64) / (nn if wterm else 1.0), device=DEV)
        lmn = torch.as_tensor(np.stack([l, m, (nn - 1.0) if wterm else 0.0 * nn]), device=DEV)
        step = max(1, (1 << 25) // len(fl))
        for r0 in range(0, uvw.shape[0], step):
            b = uvw[r0:r0 + step]
            d = b[:, :1] * lmn[0] + b[:, 1:2] * lmn[1] + b[:, 2:] * lmn[2]
            r2 = b[:, :1] ** 2 + b[:, 1:2] ** 2
            for c in range(inv.numel()):
                ph = (d * inv[c]) * (-2.0 * math.pi)
                a = amp
                if sig is not None:
                    s2 = torch.as_tensor((np.asarray(sig) * cell) ** 2, device=DEV)
                    a = amp * torch.exp((-2.0 * math.pi ** 2) * (r2 * inv[c] ** 2) * s2)
                out[r0:r0 + step, c] += torch.complex((torch.cos(ph) * a).sum(1), (torch.sin(ph) * a).sum(1))
    return out


def _points_image(pts, n, dtype):
    img = torch.zeros((n, n), dtype=dtype, device=DEV)
    dx, dy, fl = pts
    img[torch.as_tensor(n // 2 + dy), torch.as_tensor(n // 2 + dx)] = torch.as_tensor(fl, device=DEV).to(dtype)
    return img


def _noisy(case, seed, vis):
    gen = torch.Generator(device=DEV).manual_seed(int(seed) * 104729 + 5)
    noise = torch.randn(vis.shape + (2,), generator=gen, device=DEV, dtype=torch.float64)
    return (vis + 1e-2 * torch.view_as_complex(noise)).to(torch.complex128 if case["fp64"] else torch.complex64)


class State:
    """A user's program before the call: the job handles, device inputs and output buffers."""

    def __init__(self, case):
        self.case = case
        self.recs = []
        self.batch = None
        self.out = []

    def close(self):
        if self.batch is not None:
            self.batch.close()
            self.batch = None
        for r in self.recs:
            r.close()
        self.recs = []

    def __del__(self):
        self.close()


_CTX = []


def _ctx():
    if not _CTX:
        _CTX.append(rix.create(0))
    return _CTX[0]


def _rec(case, n, freq, nrow):
    return pipeline.Reconstruction(
        _ctx(), n, case["cell_as"] * ARCSEC, case["planes"], list(freq), nrow, case["parts"],
        rix.FP64 if case["fp64"] else rix.FP32,
        weighting=rix.WEIGHT_UNIFORM if case["uniform"] else rix.WEIGHT_NATURAL,
        exchange=rix.EXCHANGE_SPECTRAL if case["spectral"] else rix.EXCHANGE_IMAGE)


def _sizes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["batch"].split(",")]


def prepare(case, seed):
    st = State(case)
    op, cell = case["op"], case["cell_as"] * ARCSEC
    rdt = torch.float64 if case["fp64"] else torch.float32
    cdt = torch.complex128 if case["fp64"] else torch.complex64
    jobs = _sizes(case) if op == "major" else [(case["n"], case["nvis"])]
    for k, (n, nvis) in enumerate(jobs):
        uvw, freq, weight = _observation(case, seed + 1000 * k, nvis)
        pts, gauss = _sky(case, seed + 1000 * k, n)
        rec = _rec(case, n, freq, uvw.shape[0])
        st.recs.append(rec)
        if op in ("predict", "setup"):
            vis = torch.zeros((uvw.shape[0], len(freq)), dtype=cdt, device=DEV)
        else:
            vis = _noisy(case, seed + 1000 * k, _vis(case, uvw, freq, pts, gauss, cell))
        if op == "job":
            st.inputs = (uvw, vis, weight)
            continue
        rec.set_data(uvw, vis, weight)
        if op == "predict":
            st.image = _points_image(pts, n, rdt)
            st.out = [vis]
        elif op == "image":
            st.out = [torch.empty((n, n), dtype=rdt, device=DEV) for _ in range(rec.n_part)]
        elif op == "setup":
            st.inputs = (uvw, weight)
            # room for every sample in every partition: how many overlap depends on the observation
            ne = rec.n_part * uvw.shape[0] * len(freq)
            st.out = [torch.zeros((uvw.shape[0], len(freq)), dtype=torch.uint8, device=DEV),
                      torch.zeros(ne, dtype=torch.int32, device=DEV), torch.zeros(ne, dtype=torch.int32, device=DEV)]
            st.out += [torch.empty((2 * n, 2 * n), dtype=rdt, device=DEV) for _ in range(rec.n_part)]
        else:
            # the resident model of the cycle: the sky's points, as a first minor cycle would leave them
            img = _points_image(pts, n, rdt)
            for p in range(rec.n_part):
                rix.major_cycle(rec.job, p, rec.vis, img)
            st.out += [torch.empty((n, n), dtype=rdt, device=DEV) for _ in range(rec.n_part)]
    if op == "major":
        m = pipeline.Method("fista", iters=0)
        for rec in st.recs:
            rec.minor_all(m, torch.cuda.current_stream())
        st.batch = pipeline.BatchedMajor(_ctx(), st.recs)
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        st.batch.capture(s, residual_out=st.out)
        torch.cuda.current_stream().wait_stream(s)
    if op == "job":
        st.method = pipeline.Method(
            case["method"], scales=tuple(float(v) for v in case["scales"].split(",")) if case["scales"] else (0.0,),
            gain=0.1, niter=case["iters"], threshold=0.0, lam_rel=1e-3, iters=case["iters"], levels=case["levels"],
            dictionary="db1-8" if case["concat"] else "db4",
            schedule=(case["sched_a"], case["sched_b"]) if case["sched_a"] > 0.0 else None)
        st.out = [torch.empty((case["n"], case["n"]), dtype=rdt, device=DEV) for _ in range(case["parts"])]
    torch.cuda.synchronize()
    return st


def run(st):
    case = st.case
    op = case["op"]
    rec = st.recs[0]
    if op == "predict":
        for p in range(rec.n_part):
            rix.degrid(rec.job, p, st.image, st.out[0])
        return st.out
    if op == "image":
        for p in range(rec.n_part):
            rix.grid(rec.job, p, rec.vis, st.out[p])
        return st.out
    if op == "major":
        st.batch.replay()
        return st.out
    if op == "setup":
        rix.set_uv_partition(rec.job, st.inputs[0], st.inputs[1], None, 1.0, st.out[0])
        rix.get_sorted_entries(rec.job, st.out[1], st.out[2])
        for p in range(rec.n_part):
            rix.psf(rec.job, p, st.out[3 + p])
        return st.out
    rec.set_data(*st.inputs)
    img = rec.run(st.method, case["cycles"])
    for p in range(rec.n_part):
        rix.get_model(rec.job, p, st.out[p])
    return [img] + st.out


# -------------------------------------------------------------------- work ----
def _fft_flops(n, planes):
    """One pruned 2D transform per plane: N rows and at least N columns of length 2N."""
    return max(planes, 1) * 5.0 * 2 * n * math.log2(2 * n) * 2 * n


def work(case):
    r = 8 if case["fp64"] else 4
    op, nchan, parts = case["op"], case["nchan"], case["parts"]
    tap = 512 if case["planes"] else 64
    jobs = _sizes(case) if op == "major" else [(case["n"], case["nvis"])]
    nbytes = flops = 0.0
    for n, nvis in jobs:
        rows = nvis * 24.0 / nchan
        one = nvis * tap * 4.0 + parts * _fft_flops(n, case["planes"])       # degrid or grid
        if op == "predict":
            nbytes += n * n * r + nvis * 2 * r + rows
            flops += one
        elif op == "image":
            nbytes += parts * n * n * r + nvis * (2 * r + 4) + rows
            flops += one
        elif op == "major":
            nbytes += parts * 2 * n * n * r + nvis * (2 * r + 4) + rows
            flops += 2 * one
        else:
            psf = nvis * tap * 2.0 + parts * 4 * _fft_flops(n, case["planes"])
            if op == "setup":
                nbytes += rows + nvis * (4 + 1 + 8) + parts * 4 * n * n * r
                flops += psf
            else:
                if case["method"] == "fista":
                    nb = 8 if case["concat"] else 1
                    minor = case["iters"] * (1.5 * _fft_flops(n, 1) + nb * n * n * 80.0)
                else:
                    ns = len(case["scales"].split(","))
                    minor = case["iters"] * ns * n * n * 2.0
                nbytes += rows + nvis * (2 * r + 4) + (parts + 1) * n * n * r
                flops += psf + case["cycles"] * (2 * one + parts * minor)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------- exact ----
def _partition(case, uvw, freq, n, cell):
    """u, v, w in wavelengths per sample and each partition's member flags (every sample lies on the grid)."""
    inv = _lambdas(uvw, freq)
    u, v, w = ((uvw[:, k:k + 1] * inv).reshape(-1) for k in range(3))
    ndl = cell * n
    pu, pv = u * ndl, v * ndl
    rad = torch.sqrt(pu * pu + pv * pv)
    parts = case["parts"]
    srt = torch.sort(rad).values
    ell = [float(srt[(i * (rad.numel() - 1)) // parts]) for i in range(1, parts)]
    x = u * (cell * 2 * n) + n
    y = v * (cell * 2 * n) + n
    inside = (torch.ceil(x - 4) >= 0) & (torch.ceil(x - 4) + 8 <= 2 * n) & (torch.ceil(y - 4) >= 0) & \
             (torch.ceil(y - 4) + 8 <= 2 * n)
    masks = []
    for p in range(parts):
        ok = inside.clone()
        if p > 0:
            ok &= rad >= ell[p - 1] - 1.0
        if p < parts - 1:
            ok &= rad <= ell[p] + 1.0
        masks.append(ok)
    return u, v, w, masks


def _weights64(case, uvw, freq, weight, n, cell):
    ns = uvw.shape[0] * len(freq)
    w = torch.ones(ns, dtype=torch.float32, device=DEV) if weight is None else weight.reshape(-1)
    if not case["uniform"]:
        return w.double()
    u, v, _, masks = _partition(case, uvw, freq, n, cell)
    inside = torch.stack(masks).any(0)
    a = torch.floor(u * (cell * n) + 0.5).long()
    b = torch.floor(v * (cell * n) + 0.5).long()
    h = n // 2
    dens = torch.zeros(n * n, dtype=torch.float64, device=DEV)
    for s in (1, -1):
        i, j = h + s * a, h + s * b
        ok = inside & (i >= 0) & (i < n) & (j >= 0) & (j < n)
        dens.index_add_(0, (i * n + j)[ok], w.double()[ok])
    i, j = h + a, h + b
    ok = inside & (i >= 0) & (i < n) & (j >= 0) & (j < n)
    d = torch.where(ok, dens[((i * n + j) * ok)], torch.zeros((), dtype=torch.float64, device=DEV))
    return torch.where(d > 0, w.double() / torch.where(d > 0, d, torch.ones_like(d)), w.double()).float().double()


def _dirty(u, v, w, y, n, cell, wterm, terms):
    """Re sum_k y_k exp(2 pi i (u l + v m + w (n - 1))) / n on n x n pixels, the w-term by its Taylor series."""
    px = (torch.arange(n, dtype=torch.float64, device=DEV) - n // 2) * cell
    acc = [torch.zeros((n, n), dtype=torch.complex128, device=DEV) for _ in range(terms)]
    w0 = float(0.5 * (w.min() + w.max())) if wterm and w.numel() else 0.0
    step = max(1, (1 << 24) // n)
    for k in range(0, u.numel(), step):
        eu = torch.exp(2j * math.pi * (u[k:k + step, None] * px))
        ev = torch.exp(2j * math.pi * (v[k:k + step, None] * px)).T.contiguous()
        c = y[k:k + step].to(torch.complex128)
        for t in range(terms):
            acc[t] += ev @ (c[:, None] * eu)
            c = c * (2j * math.pi / (t + 1)) * (w[k:k + step] - w0)
    if not wterm:
        return acc[0].real
    r2 = px[None, :] ** 2 + px[:, None] ** 2
    nn = torch.sqrt(1.0 - r2)
    nm1 = -r2 / (1.0 + nn)
    img = torch.zeros_like(acc[0])
    for t in reversed(range(terms)):
        img = img * nm1 + acc[t]
    return (img * torch.exp(2j * math.pi * w0 * nm1)).real / nn


def _terms(case, w, n, cell):
    if not case["planes"]:
        return 1
    r2 = 2.0 * (0.5 * n * cell) ** 2
    a = 2.0 * math.pi * 0.5 * float(w.max() - w.min()) * r2 / (1.0 + math.sqrt(1.0 - r2))
    t, e = 1, 1.0
    while e > 1e-17:
        e *= a / t
        t += 1
    return t


def exact(case, seed):
    op, cell = case["op"], case["cell_as"] * ARCSEC
    if op == "job":
        return None
    outs = []
    for k, (n, nvis) in enumerate(_sizes(case) if op == "major" else [(case["n"], case["nvis"])]):
        uvw, freq, weight = _observation(case, seed + 1000 * k, nvis)
        pts, gauss = _sky(case, seed + 1000 * k, n)
        if op == "predict":
            ref = _vis(case, uvw, freq, pts, ((), (), (), ()), cell)
            u, v, w, masks = _partition(case, uvw, freq, n, cell)
            ref.view(-1)[~torch.stack(masks).any(0)] = 0
            return [ref]
        u, v, w, masks = _partition(case, uvw, freq, n, cell)
        side = 2 * n if op == "setup" else n
        terms = _terms(case, w, side, cell)
        if 8.0 * side * side * u.numel() * terms > 3e12:
            outs += ([None] * 3 if op == "setup" else []) + [None] * case["parts"]
            continue
        wt = _weights64(case, uvw, freq, weight, n, cell)
        if op == "setup":
            outs += [None] * 3
            y = wt.to(torch.complex128)
        else:
            vis = _noisy(case, seed + 1000 * k, _vis(case, uvw, freq, pts, gauss, cell)).to(torch.complex128)
            if op == "major":
                vis = vis - _vis(case, uvw, freq, pts, ((), (), (), ()), cell)
            y = wt * vis.reshape(-1)
        for m in masks:
            s = float(wt[m].sum())
            img = _dirty(u[m], v[m], w[m], y[m], side, cell, case["planes"] > 0, terms)
            outs.append(img / s if s > 0 else torch.zeros_like(img))
    return outs if any(o is not None for o in outs) else None
