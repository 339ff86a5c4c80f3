"""Workloads of the Pointing SelfCal library as a program runs them, for timing and for accuracy.

``listed()`` names twelve of them, ``draw(rng)`` gives others of the same
ranges, ``prepare(case, seed)`` makes what a program has in hand before the
call (inputs, contexts, plans), ``run(state)`` makes the call through the
Python binding, ``work(case)`` counts what the call cannot do without and
``exact(case, seed)`` gives its results in 64-bit torch arithmetic.

Sizes are those of the workloads in ``inputs.py`` (27 antennas of 25 m with 1
or 64 channels, 64 of 13.5 m with 16, 197 of 15 m with 16 or 128, and the
mixed batch of all three).  The observed visibilities are direct sums over
point sources seen through each antenna's shifted Airy pattern, plus thermal
noise, so they hold what a gridded model cannot reproduce, as real data do.

The library's chi^2, gradient, normal blocks and offsets are FP64 numbers
formed from FP32 evaluations: ``run`` hands them on in FP32, the accuracy
that they have.
"""
import math

import numpy as np
import torch

from paper_1709_08681_gb300 import _abi

C_LIGHT = 299792458.0
ARCSEC = math.pi / (180.0 * 3600.0)
DEG = math.pi / 180.0
ALPHA = 1.1442341324495227             # Gaussian main-lobe parameter of the uniform disk, per D_lambda
SUPPORT, OVERSAMPLE = 32, 20
LAT, DEC = 34.0 * DEG, 30.0 * DEG
SIGMA_PRIOR = 30.0 * ARCSEC
DEV = "cuda"

# Arrays and grids of the library's workloads.
ARRAYS = {
    "y27": dict(layout="y", extent=1000.0, diam=25.0, cell=8.0, n_img=2048, n_grid=2048, f=(1.0e9, 2.0e9), dt=2.0,
                sources=150, radius=1260.0),
    "y27_small": dict(layout="y", extent=1000.0, diam=25.0, cell=6.0, n_img=256, n_grid=4096, f=(1.4e9, 1.4e9),
                      dt=120.0, sources=50, radius=750.0),
    "y27_mixed": dict(layout="y", extent=1000.0, diam=25.0, cell=11.0, n_img=256, n_grid=1024, f=(1.3e9, 1.5e9),
                      dt=10.0, sources=50, radius=900.0),
    "disk64": dict(layout="disk", extent=4000.0, diam=13.5, cell=2.5, n_img=2048, n_grid=8192, f=(1.3e9, 1.5e9),
                   dt=10.0, sources=100, radius=1800.0),
    "disk197": dict(layout="disk", extent=8000.0, diam=15.0, cell=1.0, n_img=4096, n_grid=8192, f=(0.95e9, 1.76e9),
                    dt=1.0, sources=60, radius=1800.0),
    "disk197_mixed": dict(layout="disk", extent=8000.0, diam=15.0, cell=1.2, n_img=4096, n_grid=8192,
                          f=(1.3e9, 1.5e9), dt=10.0, sources=60, radius=1620.0),
}


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest use: one interval of one channel solved on its own from
        # zero offsets (psc_solve_offsets), where latency and launches count
        dict(name="solve_27ant_1ch", kind="solve", array="y27_small", n_ant=27, nt=60, nc=1),
        # one evaluation of chi^2, gradient and normals for a caller's own
        # minimiser: a five-minute interval with per-visibility weights,
        # launch shape as psc_create leaves it
        dict(name="eval_27ant_64ch", kind="eval", array="y27", n_ant=27, nt=150, nc=64, weights=True, tiling="default",
             ap="disk", bf16=False),
        # simulation or an external fit: V and the four derivative planes
        dict(name="predict_27ant_64ch", kind="predict", array="y27", n_ant=27, nt=150, nc=64, deriv=True,
             tiling="default", ap="disk", bf16=False),
        # the LM loop over an observation's four intervals in one batch, with
        # the launch shape that the autotuner settles on for this array
        dict(name="iterate_27ant_64ch", kind="batch", arrays="y27", n_ants="27", nts="150,150,150,150", nc=64,
             weights=True, tiling="flat256x2"),
        # the full-scale array, one-minute intervals at 1 s: small apertures,
        # the track kernel (two intervals of the thirty), the largest call
        dict(name="iterate_197ant_128ch", kind="batch", arrays="disk197", n_ants="197", nts="60,60", nc=128,
             weights=False, tiling="track2"),
        # intervals of uneven length on three arrays in one batch, launch
        # shapes as psc_create leaves them
        dict(name="iterate_mixed", kind="batch", arrays="y27_mixed,disk64,disk197_mixed,disk64,y27_mixed",
             n_ants="27,64,197,64,27", nts="411,173,77,59,38", nc=16, weights=False, tiling="default"),
        # large pointing offsets: the exact kernel of two shifted disks, in
        # its benchmark shape
        dict(name="exact_27ant_64ch", kind="eval", array="y27", n_ant=27, nt=150, nc=64, weights=False,
             tiling="flat256x1", model="exact", ap="disk", bf16=False),
        # a long interval with its residual w (a stack of grids), in its
        # benchmark shape
        dict(name="stack_27ant_64ch", kind="eval", array="y27", n_ant=27, nt=600, nc=64, weights=False,
             tiling="flat128x1", model="stack", planes=33, ap="disk", bf16=False),
        # the learned initial estimate of a batch of intervals: features of
        # every antenna on two of the 60 samples, then the network
        dict(name="learned_init_64ant", kind="learned", n_geom=8, n_int=128, nt=60, nc=16, n_ant=64, stride=30),
        # its training: loss and gradient of one minibatch
        dict(name="mlp_grad_1024", kind="mlp_grad", batch=1024),
        # the model grid of an image, padded four times (once per model)
        dict(name="grid_2048_to_8192", kind="grid", n_img=2048, n_grid=8192, cell=2.5, sources=2000),
        # the model grid of point components (once per interval with W-snapshots)
        dict(name="grid_2000_components", kind="components", n_comp=2000, n_grid=2048, cell=8.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _nt(rng, n_ant, nc, lo, hi, most):
    """Time steps of an interval with at most `most` visibilities."""
    top = max(1, min(hi, int(most // (n_ant * (n_ant - 1) // 2 * nc))))
    return _log(rng, min(lo, top), top)


def draw(rng):
    kind = rng.choice(["solve", "eval", "predict", "iterate", "track", "mixed", "exact", "stack", "learned", "mlp_grad",
                       "grid", "components"])
    if kind == "solve":
        n_ant = rng.randint(5, 64)
        nc = rng.randint(1, 8)
        return dict(kind="solve", array="y27_small" if nc == 1 else "y27", n_ant=n_ant, nt=_nt(rng, n_ant, nc, 20, 150, 2e6),
                    nc=nc)
    if kind in ("eval", "predict"):
        array = rng.choice(["y27", "y27_mixed", "disk64", "disk197"])
        n_ant = _log(rng, 4, 197 if array == "disk197" else 64)
        nc = _log(rng, 1, 128)
        c = dict(kind=kind, array=array, n_ant=n_ant, nt=_nt(rng, n_ant, nc, 1, 600, 1.2e7), nc=nc,
                 tiling=rng.choice(["default", "default", "flat256x1", "rect75x3x1"]),
                 ap="gauss" if rng.random() < 0.15 else "disk", bf16=rng.random() < 0.2)
        if kind == "eval":
            c["weights"] = rng.random() < 0.5
        else:
            c["deriv"] = rng.random() < 0.5
        if c["tiling"].startswith("flat") and c["nt"] < 40:
            c["tiling"] = "default"
        return c
    if kind == "iterate":
        n_ant, n_int = rng.randint(8, 40), rng.randint(1, 6)
        nc = _log(rng, 3, 64)
        nts = [max(90, _nt(rng, n_ant, nc, 90, 300, 6e6)) for _ in range(n_int)]
        return dict(kind="batch", arrays="y27", n_ants=str(n_ant), nts=",".join(map(str, nts)), nc=nc,
                    weights=rng.random() < 0.5, tiling=rng.choice(["flat256x2", "flat192x2", "flat128x1", "default"]))
    if kind == "track":
        n_ant, n_int = _log(rng, 24, 197), rng.randint(1, 2)
        nc = _log(rng, 8, 128)
        nts = [_nt(rng, n_ant, nc, 17, 130, 1.4e8) for _ in range(n_int)]
        return dict(kind="batch", arrays="disk197", n_ants=str(n_ant), nts=",".join(map(str, nts)), nc=nc,
                    weights=rng.random() < 0.3, tiling=rng.choice(["track1", "track2", "track2"]))
    if kind == "mixed":
        n_int = rng.randint(2, 8)
        arrays = [rng.choice(["y27_mixed", "disk64", "disk197_mixed"]) for _ in range(n_int)]
        n_ants = [{"y27_mixed": 27, "disk64": 64, "disk197_mixed": 197}[a] for a in arrays]
        nts = [_nt(rng, n, 16, 30, 600, 2.2e7) for n in n_ants]
        return dict(kind="batch", arrays=",".join(arrays), n_ants=",".join(map(str, n_ants)),
                    nts=",".join(map(str, nts)), nc=16, weights=False, tiling=rng.choice(["default", "track1"]))
    if kind == "exact":
        n_ant, nc = rng.randint(5, 36), _log(rng, 1, 64)
        return dict(kind="eval", array="y27", n_ant=n_ant, nt=max(45, _nt(rng, n_ant, nc, 45, 300, 4e6)), nc=nc,
                    weights=rng.random() < 0.5, tiling=rng.choice(["flat256x1", "default"]), model="exact", ap="disk",
                    bf16=False)
    if kind == "stack":
        n_ant, nc = rng.randint(6, 36), _log(rng, 2, 64)
        return dict(kind="eval", array="y27", n_ant=n_ant, nt=max(60, _nt(rng, n_ant, nc, 60, 900, 1.3e7)), nc=nc,
                    weights=rng.random() < 0.5, tiling=rng.choice(["flat128x1", "default"]), model="stack",
                    planes=rng.randint(3, 40), ap="disk", bf16=False)
    if kind == "learned":
        return dict(kind="learned", n_geom=rng.randint(1, 8), n_int=_log(rng, 4, 128), nt=60, nc=rng.choice([4, 16, 16]),
                    n_ant=rng.randint(12, 64), stride=rng.choice([15, 20, 30, 60]))
    if kind == "mlp_grad":
        return dict(kind="mlp_grad", batch=_log(rng, 1, 4096))
    if kind == "grid":
        n_img = 2 * rng.randint(64, 1024) if rng.random() < 0.4 else 8 * rng.randint(16, 256)
        if n_img % 8:
            n_img = min(n_img, 700)
        return dict(kind="grid", n_img=n_img, n_grid=n_img * rng.choice([1, 2, 4]), cell=2.5,
                    sources=_log(rng, 50, 5000))
    return dict(kind="components", n_comp=_log(rng, 1, 4000), n_grid=2 * rng.randint(128, 1024), cell=8.0)


# ---------------------------------------------------------------- inputs

def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000 + stream)
    return g


def _layout(layout, n_ant, extent, rng):
    """East and north positions (m) of a Y array or a centrally concentrated random disk."""
    if layout == "y":
        arm = np.arange(n_ant) % 3
        r = extent * rng.uniform(0.02, 1.0, n_ant)
        az = (5.0 + 120.0 * arm) * DEG
        return np.stack([r * np.sin(az), r * np.cos(az)], 1)
    n_in = n_ant // 2
    r = extent * np.concatenate([0.2 * np.sqrt(rng.uniform(0, 1, n_in)), np.sqrt(0.04 + 0.96 * rng.uniform(0, 1, n_ant - n_in))])
    th = rng.uniform(0, 2 * math.pi, n_ant)
    return np.stack([r * np.sin(th), r * np.cos(th)], 1)


class Sky:
    """An array recipe's sky (a point-source list) and its model grid."""

    def __init__(self, rec, seed, stream):
        rng = np.random.default_rng([int(seed), stream])
        k = rec["sources"]
        r = rec["radius"] * ARCSEC * np.sqrt(rng.uniform(0, 1, k))
        r = np.minimum(r, 0.49 * rec["n_img"] * rec["cell"] * ARCSEC)
        th = rng.uniform(0, 2 * math.pi, k)
        cell = rec["cell"] * ARCSEC
        l = np.rint(r * np.sin(th) / cell / 1.5) * cell
        m = np.rint(r * np.cos(th) / cell / 1.5) * cell
        s = (1e-2 ** -0.5 + rng.uniform(0, 1, k) * (1.0 - 1e-2 ** -0.5)) ** -2.0     # p(S) ~ S^-1.5 on [0.01, 1] Jy
        self.lms = torch.from_numpy(np.stack([l, m, s], 1)).to(DEV)
        self.n_grid, self.cell = rec["n_grid"], cell
        self.du = 1.0 / (self.n_grid * cell)

    def grid(self, lms=None, flux=None):
        """sum_k S_k exp(2 pi i (u l_k + v m_k)) on the grid, complex64 [Ng][Ng]."""
        lms = self.lms if lms is None else lms
        flux = lms[:, 2].to(torch.complex128) if flux is None else flux
        u = (torch.arange(self.n_grid, dtype=torch.float64, device=DEV) - self.n_grid // 2) * self.du
        a = torch.polar(torch.ones((), dtype=torch.float64, device=DEV), 2 * math.pi * (u[:, None] * lms[None, :, 0]))
        b = torch.polar(torch.ones((), dtype=torch.float64, device=DEV), 2 * math.pi * (u[:, None] * lms[None, :, 1]))
        return b.to(torch.complex64) @ (a * flux[None, :]).to(torch.complex64).T


class Obs:
    """One solution interval's inputs: antennas, uvw, channels, true offsets and observed data."""

    def __init__(self, rec, n_ant, nt, nc, sky, seed, stream, weights=False, w_term=False, sigma=20.0, hour=None,
                 layout_stream=None, data=True, noise=1e-3):
        rng = np.random.default_rng([int(seed), 7, stream])
        lay = rng if layout_stream is None else np.random.default_rng([int(seed), 9, layout_stream])
        self.n_ant, self.nt, self.nc, self.sky, self.diam = n_ant, nt, nc, sky, rec["diam"]
        self.n_bl = n_ant * (n_ant - 1) // 2
        pos = _layout(rec["layout"], n_ant, rec["extent"], lay)
        f0, f1 = rec["f"]
        self.freq = f0 + (np.arange(nc) + 0.5) * (f1 - f0) / nc
        hour = rng.uniform(-2.0, 2.0) if hour is None else hour
        ha = torch.from_numpy(hour * 15.0 * DEG + (np.arange(nt) - (nt - 1) / 2) * rec["dt"] / 3600.0 * 15.0 * DEG).to(DEV)
        e, n = (torch.from_numpy(np.ascontiguousarray(pos[:, k])).to(DEV) for k in (0, 1))
        x, y, z = -math.sin(LAT) * n, e, math.cos(LAT) * n
        sh, ch = torch.sin(ha)[:, None], torch.cos(ha)[:, None]
        sd, cd = math.sin(DEC), math.cos(DEC)
        self.ant = torch.stack([sh * x + ch * y, -sd * ch * x + sd * sh * y + cd * z, cd * ch * x - cd * sh * y + sd * z], -1)
        i, j = torch.triu_indices(n_ant, n_ant, 1, device=DEV)
        self.i, self.j = i, j
        self.uvw = (self.ant[:, j] - self.ant[:, i]).contiguous()
        self.lm_true = rng.normal(0.0, sigma * ARCSEC, (n_ant, 2))
        self.noise = noise
        self.w_scale = 1.0 / noise ** 2
        self.w = None
        if weights:
            self.w = torch.empty((nt, self.n_bl, nc), device=DEV)
            self.w.uniform_(0.2, 1.8, generator=_gen(seed, 300 + stream))
        self.vis = self._observe(_gen(seed, 200 + stream), w_term) if data else None

    def _observe(self, gen, w_term):
        k = self.sky.lms.shape[0]
        l, m, s = self.sky.lms[:, 0], self.sky.lms[:, 1], self.sky.lms[:, 2]
        p = torch.from_numpy(self.lm_true).to(DEV)
        nu = torch.from_numpy(self.freq / C_LIGHT).to(DEV)
        rho = torch.hypot(l[None] - p[:, :1], m[None] - p[:, 1:])
        x = math.pi * self.diam * nu[:, None, None] * rho[None] + 1e-9
        beam = (2.0 * torch.special.bessel_j1(x) / x * torch.sqrt(s)).to(torch.float32)      # [nc][n_ant][k]
        path = self.ant[..., :1] * l + self.ant[..., 1:2] * m
        if w_term:
            path = path + self.ant[..., 2:] * (torch.sqrt(1.0 - l * l - m * m) - 1.0)
        out = torch.empty((self.nt, self.n_bl, self.nc), dtype=torch.complex64, device=DEV)
        step = max(1, int(2e7 // (self.nc * self.n_ant * max(k, self.n_ant))))
        for t in range(0, self.nt, step):
            ph = nu[:, None, None] * path[t:t + step, None]
            ph = (2 * math.pi * (ph - torch.round(ph))).to(torch.float32)
            e = torch.polar(beam.expand_as(ph).contiguous(), ph)
            v = e.conj().resolve_conj() @ e.transpose(-1, -2)
            out[t:t + step] = v[:, :, self.i, self.j].transpose(1, 2)
        noise = torch.randn(out.shape + (2,), generator=gen, device=DEV)
        out += torch.view_as_complex(noise) * self.noise
        return out

    def context(self, grid, ap="disk", stream=None):
        s = self.sky
        return _abi.Context(self.n_ant, self.nt, self.nc, self.uvw, self.freq, ap, self.diam, ALPHA, 1, s.n_grid, s.n_grid,
                            s.cell, SUPPORT, OVERSAMPLE, grid, stream)


def _set_tiling(ctx, tiling):
    if tiling.startswith("flat"):
        items, kv = tiling[4:].split("x")
        ctx.psc_set_flat_tiling(int(items), int(kv))
    elif tiling.startswith("rect"):
        ctx.psc_set_tiling(*(int(x) for x in tiling[4:].split("x")))
    elif tiling.startswith("track"):
        ctx.psc_set_track_tiling(int(tiling[5:]))


def _stack(case, obs):
    """The residual-w stack of an interval: plane fit, moved components, planes and their spacing."""
    s, uvw = obs.sky, obs.uvw.reshape(-1, 3)
    uu, uv, vv, uw, vw = (float((uvw[:, p] * uvw[:, q]).sum()) for p, q in ((0, 0), (0, 1), (1, 1), (0, 2), (1, 2)))
    det = uu * vv - uv * uv
    a, b = (uw * vv - vw * uv) / det, (vw * uu - uw * uv) / det
    l, m, flux = s.lms[:, 0], s.lms[:, 1], s.lms[:, 2]
    nm1 = torch.sqrt(1.0 - l * l - m * m) - 1.0
    lms = torch.stack([l + a * nm1, m + b * nm1, flux], 1)
    r = uvw[:, 2] - a * uvw[:, 0] - b * uvw[:, 1]
    lo, hi = (float(f(r)) for f in (torch.min, torch.max))
    f0, f1 = float(obs.freq.min()) / C_LIGHT, float(obs.freq.max()) / C_LIGHT
    w_lo, w_hi = min(lo * f0, lo * f1), max(hi * f0, hi * f1)
    dw = (w_hi - w_lo) * (1 + 1e-6) / (case["planes"] - 1)
    w0 = w_lo - 0.25e-6 * (w_hi - w_lo)
    planes = torch.empty((case["planes"], s.n_grid, s.n_grid), dtype=torch.complex64, device=DEV)
    for p in range(case["planes"]):
        planes[p] = s.grid(lms, torch.polar(flux, 2 * math.pi * (w0 + p * dw) * nm1))
    return dict(planes=planes, w0=w0, dw=dw, a=a, b=b)


def _batch_inputs(case, seed):
    """The intervals of a batch, with one sky and grid per array type."""
    nts = [int(x) for x in case["nts"].split(",")]
    arrays, n_ants = case["arrays"].split(","), [int(x) for x in case["n_ants"].split(",")]
    arrays, n_ants = (v * len(nts) if len(v) == 1 else v for v in (arrays, n_ants))
    skies, grids, obs = {}, {}, []
    for k, (a, n, nt) in enumerate(zip(arrays, n_ants, nts)):
        if a not in skies:
            skies[a] = Sky(ARRAYS[a], seed, 1 + len(skies))
            grids[a] = skies[a].grid()
        obs.append(Obs(ARRAYS[a], n, nt, case["nc"], skies[a], seed, k, case["weights"], sigma=30.0,
                       layout_stream=sorted(skies).index(a)))
    return obs, [grids[a] for a in arrays]


def _one_input(case, seed):
    rec = ARRAYS[case["array"]]
    sky = Sky(rec, seed, 1)
    stack = case.get("model") == "stack"
    return Obs(rec, case["n_ant"], case["nt"], case["nc"], sky, seed, 0, case.get("weights", False), w_term=stack,
               sigma=60.0 if case.get("model") == "exact" else 20.0, data=case["kind"] != "predict")


def _half(lm):
    """Offsets in the middle of a solve."""
    return np.ascontiguousarray(0.6 * lm)


def _learned_inputs(case, seed):
    rec = ARRAYS["disk64"]
    sky = Sky(rec, seed, 1)
    hours = np.linspace(-3.0, 3.0, case["n_geom"])
    obs = [Obs(rec, case["n_ant"], case["nt"], case["nc"], sky, seed, k, sigma=30.0, hour=float(hours[k % case["n_geom"]]),
               layout_stream=1, noise=5e-4) for k in range(case["n_int"])]
    return sky, obs


def _network(seed):
    """He-initialised weights, small biases, an input standardisation: the flat parameter vector."""
    rng = np.random.default_rng([int(seed), 31])
    parts = []
    for i, o in ((52, 256), (256, 256), (256, 256), (256, 2)):
        parts += [rng.normal(0, math.sqrt(2.0 / i), i * o), rng.normal(0, 0.02, o)]
    mu = np.concatenate([np.zeros(2), 0.9 * np.ones(25), 0.05 * np.ones(25)])
    sd = np.concatenate([np.ones(2), 0.15 * np.ones(25), 0.1 * np.ones(25)])
    return np.concatenate(parts + [mu, sd]).astype(np.float32)


def _minibatch(case, seed):
    p = torch.from_numpy(_network(seed)[-104:]).to(DEV)
    x = p[:52] + p[52:] * torch.randn((case["batch"], 52), generator=_gen(seed, 41), device=DEV)
    return x.contiguous(), torch.randn((case["batch"], 2), generator=_gen(seed, 42), device=DEV)


def _image(case, seed):
    rng = np.random.default_rng([int(seed), 51])
    n, k = case["n_img"], case["sources"]
    img = np.zeros((n, n))
    at = rng.integers(n // 8, n - n // 8, (k, 2))
    np.add.at(img, (at[:, 0], at[:, 1]), (1e-4 ** -0.5 + rng.uniform(0, 1, k) * (1 - 1e-4 ** -0.5)) ** -2.0)
    return torch.from_numpy(img.astype(np.float32)).to(DEV)


def _components(case, seed):
    rng = np.random.default_rng([int(seed), 52])
    k = case["n_comp"]
    lm = rng.uniform(-1, 1, (k, 2)) * 0.3 * case["n_grid"] * case["cell"] * ARCSEC
    return np.ascontiguousarray(np.concatenate([lm, (1e-4 ** -0.5 + rng.uniform(0, 1, (k, 1)) * (1 - 1e-4 ** -0.5)) ** -2.0], 1))


# ---------------------------------------------------------------- prepare and run

def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("solve", "eval", "predict"):
        obs = _one_input(case, seed)
        grid = obs.sky.grid()
        ctx = obs.context(grid, case.get("ap", "disk"))
        if case.get("model") == "exact":
            ctx.psc_set_kernel_model(_abi.PSC_KERNEL_EXACT_DISK)
        elif case.get("model") == "stack":
            sk = _stack(case, obs)
            ctx.psc_set_wstack(sk["planes"], case["planes"], sk["w0"], sk["dw"], sk["a"], sk["b"])
            st["stack"] = sk
        if case.get("bf16"):
            ctx.psc_set_grid_precision(_abi.PSC_GRID_BF16)
        _set_tiling(ctx, case.get("tiling", "default"))
        st.update(obs=obs, grid=grid, ctx=ctx, lm=_half(obs.lm_true))
        if kind == "predict":
            shape = (obs.nt, obs.n_bl, obs.nc)
            st["vis"] = torch.empty(shape, dtype=torch.complex64, device=DEV)
            st["dvis"] = torch.empty((4,) + shape, dtype=torch.complex64, device=DEV) if case["deriv"] else None
            st["lm_dev"] = torch.from_numpy(st["lm"]).to(DEV)
    elif kind == "batch":
        obs, grids = _batch_inputs(case, seed)
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        ctxs = [o.context(g, stream=stream) for o, g in zip(obs, grids)]
        for c in ctxs:
            _set_tiling(c, case["tiling"])
        batch = _abi.Batch(ctxs, [o.vis for o in obs], [o.w for o in obs] if case["weights"] else None,
                           [o.w_scale for o in obs], stream)
        batch.psc_batch_begin([np.zeros((o.n_ant, 2)) for o in obs])
        st.update(obs=obs, grids=grids, ctxs=ctxs, batch=batch, stream=stream)
    elif kind == "learned":
        sky, obs = _learned_inputs(case, seed)
        grid = sky.grid()
        ctxs = [o.context(grid) for o in obs[:case["n_geom"]]]
        pairs = [ctxs[k % len(ctxs)] for k in range(case["n_int"])]
        rows = case["n_int"] * case["n_ant"]
        net = _abi.Mlp(rows)
        net.psc_mlp_set_params(_network(seed))
        work = torch.empty(_abi.psc_features_batch_work(pairs, case["stride"]), dtype=torch.uint8, device=DEV)
        st.update(obs=obs, grid=grid, ctxs=ctxs, pairs=pairs, net=net, work=work,
                  feat=torch.empty((rows, 52), dtype=torch.float32, device=DEV),
                  y=torch.empty((rows, 2), dtype=torch.float32, device=DEV))
    elif kind == "mlp_grad":
        x, t = _minibatch(case, seed)
        net = _abi.Mlp(case["batch"])
        net.psc_mlp_set_params(_network(seed))
        st.update(x=x, t=t, net=net)
    elif kind == "grid":
        st.update(img=_image(case, seed), out=torch.empty((case["n_grid"],) * 2, dtype=torch.complex64, device=DEV))
    elif kind == "components":
        st.update(comp=_components(case, seed), out=torch.empty((case["n_grid"],) * 2, dtype=torch.complex64, device=DEV))
    torch.cuda.synchronize()
    return st


def _f32(*arrays):
    return [np.asarray(a, dtype=np.float32) for a in arrays]


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "solve":
        lm, rep = st["ctx"].psc_solve_offsets(st["obs"].vis, None, st["obs"].w_scale)
        return _f32(lm / ARCSEC, rep.chi2)
    if kind == "eval":
        o = st["obs"]
        return _f32(*st["ctx"].psc_residual_grad(st["lm"], o.vis, o.w, o.w_scale, cross=True))
    if kind == "predict":
        st["ctx"].psc_predict_dev(st["lm_dev"], st["vis"], st["dvis"])
        return [st["vis"]] if st["dvis"] is None else [st["vis"], st["dvis"]]
    if kind == "batch":
        b = st["batch"]
        b.psc_batch_restart()
        b.psc_batch_iterate(2)
        lms, reps = b.psc_batch_end()
        return _f32(*[lm / ARCSEC for lm in lms]) + _f32([r.chi2 for r in reps])
    if kind == "learned":
        o = st["obs"]
        _abi.psc_features_batch(st["pairs"], [x.vis for x in o], [x.w_scale for x in o], SIGMA_PRIOR, case["stride"],
                                st["work"], st["feat"])
        st["net"].psc_mlp_forward(st["feat"], st["y"])
        return [st["feat"], st["y"]]
    if kind == "mlp_grad":
        loss, g = st["net"].psc_mlp_grad(st["x"], st["t"])
        return [np.float32(loss), g]
    if kind == "grid":
        _abi.psc_model_grid(case["n_img"], case["n_grid"], case["cell"] * ARCSEC, SUPPORT, OVERSAMPLE, st["img"], st["out"])
        return st["out"]
    _abi.psc_model_grid_components(st["comp"], case["n_grid"], case["cell"] * ARCSEC, st["out"])
    return st["out"]


# ---------------------------------------------------------------- work

def _taps(rec, nc, ap="disk"):
    """Non-zero taps of one visibility of every channel, summed over the channels."""
    f0, f1 = rec["f"]
    f = f0 + (np.arange(nc) + 0.5) * (f1 - f0) / nc
    du = 1.0 / (rec["n_grid"] * rec["cell"] * ARCSEC)
    if ap == "gauss":
        return nc * SUPPORT ** 2
    return float(np.sum(math.pi * (rec["diam"] * f / C_LIGHT / du) ** 2))


def _eval_work(rec, n_ant, nt, nc, ap="disk", weights=False, out_bytes=0, per_tap=15):
    n_bl = n_ant * (n_ant - 1) // 2
    vis = nt * n_bl * nc
    return (vis * (8 + (4 if weights else 0)) + nt * n_bl * 16 if not out_bytes else vis * out_bytes + nt * n_bl * 16,
            nt * n_bl * _taps(rec, nc, ap) * per_tap + 100.0 * vis)


def work(case):
    """Per pass: inputs read once and outputs written once; a non-zero tap costs 15 FP32 operations (61 with
    the exact disk kernel, 19 with two planes, about 70 with the 25 trial offsets)."""
    kind = case["kind"]
    if kind in ("solve", "eval", "predict"):
        rec = ARRAYS[case["array"]]
        per = {"exact": 61, "stack": 19}.get(case.get("model"), 15)
        evals = 5 if kind == "solve" else 1
        out = 8 * (5 if case.get("deriv") else 1) if kind == "predict" else 0
        b, f = _eval_work(rec, case["n_ant"], case["nt"], case["nc"], case.get("ap", "disk"), case.get("weights", False), out, per)
        return dict(bytes=b * evals, flops=f * evals)
    if kind == "batch":
        nts = [int(x) for x in case["nts"].split(",")]
        arrays, n_ants = case["arrays"].split(","), [int(x) for x in case["n_ants"].split(",")]
        arrays, n_ants = (v * len(nts) if len(v) == 1 else v for v in (arrays, n_ants))
        tot = np.sum([_eval_work(ARRAYS[a], n, nt, case["nc"], weights=case["weights"]) for a, n, nt in zip(arrays, n_ants, nts)], axis=0)
        return dict(bytes=2 * float(tot[0]), flops=2 * float(tot[1]))
    if kind == "learned":
        kept = -(-case["nt"] // case["stride"])
        b, f = _eval_work(ARRAYS["disk64"], case["n_ant"], kept, case["nc"], per_tap=70)
        rows = case["n_int"] * case["n_ant"]
        net = 52 * 256 + 2 * 256 * 256 + 512
        return dict(bytes=b * case["n_int"] + rows * 54 * 4 + 4 * net, flops=f * case["n_int"] + 2.0 * rows * net)
    if kind == "mlp_grad":
        net = 52 * 256 + 2 * 256 * 256 + 512
        return dict(bytes=case["batch"] * 54 * 4 + 8 * net, flops=6.0 * case["batch"] * net)
    if kind == "grid":
        n, g = case["n_img"], case["n_grid"]
        return dict(bytes=4.0 * n * n + 8.0 * g * g, flops=4.0 * n * n * g + 8.0 * n * g * g)
    return dict(bytes=24.0 * case["n_comp"] + 8.0 * case["n_grid"] ** 2, flops=8.0 * case["n_comp"] * case["n_grid"] ** 2)


# ---------------------------------------------------------------- the same in 64 bits

def _aperture(ap, diam, f, du, q):
    """A°(q) du^2 of a uniform disk (its autocorrelation over its area squared) or of the Gaussian pattern."""
    dl = diam * f / C_LIGHT
    if ap == "gauss":
        a2 = (ALPHA * dl) ** 2
        return math.pi / (2 * a2) * np.exp(-(math.pi * q) ** 2 / (2 * a2)) * du * du
    r = dl / 2
    x = np.minimum(q / dl, 1.0)
    return np.where(q < dl, 2 * r * r * np.arccos(x) - 0.5 * q * np.sqrt(np.maximum(dl * dl - q * q, 0)), 0.0) / (math.pi * r * r) ** 2 * du * du


def _reach(ap, diam, f, du):
    return SUPPORT / 2 * math.sqrt(2) if ap == "gauss" else diam * f / C_LIGHT / du


def _lens_moments(diam, f, du, n):
    """Moments M_pq = int w_par^p w_perp^q over the overlap of two disks n du / ov apart, p + q = 0, 2, 4, 6, over the disks' area squared."""
    r = 0.5 * diam * f / C_LIGHT
    rho = np.minimum(np.arange(n) * du / OVERSAMPLE, 2 * r)
    node, wt = np.polynomial.legendre.leggauss(48)
    th0 = np.arccos(rho / (2 * r))[:, None]
    th, wt = 0.5 * th0 * (node + 1), 0.5 * th0 * wt
    par, h = r * np.cos(th) - rho[:, None] / 2, r * np.sin(th)
    out = {(p, q): np.sum(wt * par ** p * h ** (q + 2), 1) * 4 / (q + 1) * du * du / (math.pi * r * r) ** 2
           for p in (0, 2, 4, 6) for q in (0, 2, 4, 6) if p + q <= 6}
    return {k: torch.from_numpy(v).to(DEV) for k, v in out.items()}


def _lerp(tab, t):
    k = torch.floor(t).long()
    inside = k + 1 < tab.numel()
    k = torch.where(inside, k, 0)
    f = t - torch.floor(t)
    return torch.where(inside, (1 - f) * tab[k] + f * tab[k + 1], 0.0)


def _degrid(obs, c, grid, rows, ap="disk", bf16=False, stack=None, stencil=False, exact_lm=None, L=None, M=None):
    """Sums over one channel's taps for the visibilities uvw[rows] (all times and baselines by default):
    T = sum A G, Tu, Tv = its moments in the tap offset (wavelengths), with the ramp exp(i pi (du L + dv M)), and, with
    exact_lm = (dl, dm), the sums Gl, Gm that carry the offset difference's derivatives.  stencil: T[5][5] over L = a sigma, M = b sigma."""
    f, du, ng = obs.freq[c], obs.sky.du, obs.sky.n_grid
    uvw = obs.uvw[rows].reshape(-1, 3)
    reach = _reach(ap, obs.diam, f, du)
    n_tab = int(math.floor(OVERSAMPLE * reach)) + 2
    h = min(SUPPORT // 2, int(math.ceil(reach)) + 1)
    if exact_lm is None:
        tab = torch.from_numpy(_aperture(ap, obs.diam, f, du, np.arange(n_tab) * du / OVERSAMPLE)).to(DEV)
    else:
        mom = _lens_moments(obs.diam, f, du, n_tab)
        g1, g2, g3 = (s * (2 * math.pi) ** (2 * n) / math.factorial(2 * n) for n, s in ((1, -1), (2, 1), (3, -1)))
    x, y = (uvw[:, k] * (f / C_LIGHT / du) + ng // 2 for k in (0, 1))
    x0, y0 = torch.floor(x), torch.floor(y)
    if stack is not None:
        q = (uvw[:, 2] - stack["a"] * uvw[:, 0] - stack["b"] * uvw[:, 1]) * (f / C_LIGHT) / stack["dw"] - stack["w0"] / stack["dw"]
        p = torch.clamp(torch.floor(q), 0, stack["planes"].shape[0] - 2)
        wf, p = (q - p)[:, None], p.long()[:, None] * ng * ng
        flat = stack["planes"].reshape(-1)
    else:
        flat = grid.reshape(-1)
    cols = torch.arange(-h + 1, h + 1, device=DEV)
    dx = (x - x0)[:, None] - cols
    gx = x0.long()[:, None] + cols
    in_x = (gx >= 0) & (gx < ng)
    one = torch.ones((), dtype=torch.float64, device=DEV)
    if stencil:
        ph = math.pi * du * SIGMA_PRIOR
        zx = [torch.polar(one, ph * a * dx) for a in range(-2, 3)]
        T = torch.zeros((5, 5, x.numel()), dtype=torch.complex128, device=DEV)
    else:
        ex = torch.polar(one, math.pi * du * dx * L[:, None])
        T = torch.zeros(x.numel(), dtype=torch.complex128, device=DEV)
    zero = torch.zeros(x.numel(), dtype=torch.complex128, device=DEV)
    Tu, Tv, Gl, Gm = zero.clone(), zero.clone(), zero.clone(), zero.clone()
    for b in range(-h + 1, h + 1):
        dy = (y - y0) - b
        gy = y0.long() + b
        ok = in_x & ((gy >= 0) & (gy < ng))[:, None]
        at = torch.where(ok, gy[:, None] * ng + gx, 0)
        if stack is not None:
            g = (1 - wf) * flat[p + at] + wf * flat[p + ng * ng + at]
        else:
            g = flat[at]
            if bf16:
                g = torch.complex(g.real.bfloat16().float(), g.imag.bfloat16().float())
        g = torch.where(ok, g.to(torch.complex128), 0)
        r2 = dx * dx + (dy * dy)[:, None]
        t = torch.sqrt(r2) * OVERSAMPLE
        if exact_lm is None:
            ag = _lerp(tab, t) * g
        else:
            dl, dm = (v[:, None] for v in exact_lm)
            m = {k: _lerp(v, t) for k, v in mom.items()}
            rat = (dl * dx + dm * dy[:, None]) / torch.clamp(r2, min=1e-30)
            A = (dl * dx + dm * dy[:, None]) * rat
            B = dl * dl + dm * dm - A
            O = (m[0, 0] + g1 * (A * m[2, 0] + B * m[0, 2]) + g2 * (A * A * m[4, 0] + 6 * A * B * m[2, 2] + B * B * m[0, 4])
                 + g3 * (A ** 3 * m[6, 0] + 15 * A * A * B * m[4, 2] + 15 * A * B * B * m[2, 4] + B ** 3 * m[0, 6]))
            OA = g1 * m[2, 0] + g2 * (2 * A * m[4, 0] + 6 * B * m[2, 2]) + g3 * (3 * A * A * m[6, 0] + 30 * A * B * m[4, 2] + 15 * B * B * m[2, 4])
            OB = g1 * m[0, 2] + g2 * (6 * A * m[2, 2] + 2 * B * m[0, 4]) + g3 * (15 * A * A * m[4, 2] + 30 * A * B * m[2, 4] + 3 * B * B * m[0, 6])
            W = (OA - OB) * rat
            ey = torch.polar(one, math.pi * du * dy * M)
            Gl += (2 * (W * dx + OB * dl) * g * ex).sum(1) * ey
            Gm += (2 * (W * dy[:, None] + OB * dm) * g * ex).sum(1) * ey
            ag = O * g
        if stencil:
            R = torch.stack([(ag * z).sum(1) for z in zx])
            for k in range(5):
                T[k] += R * torch.polar(one, ph * (k - 2) * dy)
            Tu += (ag * dx).sum(1)
            Tv += R[2] * dy
        else:
            ag = ag * ex
            ey = torch.polar(one, math.pi * du * dy * M)
            P = ag.sum(1) * ey
            T += P
            Tu += (ag * dx).sum(1) * ey
            Tv += P * dy
    return T, Tu * du, Tv * du, Gl, Gm


def _model(obs, c, grid, lm, **how):
    """V and dV/d(l_i, m_i, l_j, m_j) of one channel, [nt * n_bl]."""
    ex = how.pop("exact", False)
    p = torch.from_numpy(lm).to(DEV)
    s, d = p[obs.i] + p[obs.j], p[obs.i] - p[obs.j]
    L, M, dl, dm = (v.repeat(obs.nt) for v in (s[:, 0], s[:, 1], d[:, 0], d[:, 1]))
    out = []
    n, chunk = obs.nt, max(1, int(3e6 // (obs.n_bl * 20)))
    for t in range(0, n, chunk):
        k = slice(t * obs.n_bl, min(n, t + chunk) * obs.n_bl)
        T, Tu, Tv, Gl, Gm = _degrid(obs, c, grid, slice(t, t + chunk), L=L[k], M=M[k], exact_lm=(dl[k], dm[k]) if ex else None, **how)
        ip = 1j * math.pi
        if ex:
            out.append(torch.stack([T, ip * Tu + Gl, ip * Tv + Gm, ip * Tu - Gl, ip * Tv - Gm]))
            continue
        a2 = (ALPHA * obs.diam * obs.freq[c] / C_LIGHT) ** 2
        D = torch.exp(-0.5 * a2 * (dl[k] ** 2 + dm[k] ** 2))
        el, em = -dl[k] * a2, -dm[k] * a2
        out.append(D * torch.stack([T, el * T + ip * Tu, em * T + ip * Tv, -el * T + ip * Tu, -em * T + ip * Tv]))
    return torch.cat(out, 1)


def _evaluate(obs, grid, lm, **how):
    """chi^2, gradient [n][2], normal blocks [n][3] and cross blocks [n_bl][4]."""
    sums = torch.zeros((15, obs.n_bl), dtype=torch.float64, device=DEV)
    for c in range(obs.nc):
        V = _model(obs, c, grid, lm, **how)
        w = torch.full((obs.nt * obs.n_bl,), obs.w_scale, dtype=torch.float64, device=DEV)
        if obs.w is not None:
            w = w * obs.w[:, :, c].reshape(-1).double()
        R = obs.vis[:, :, c].reshape(-1).to(torch.complex128) - V[0]
        re = lambda a, b: (w * (a.conj() * b).real).reshape(obs.nt, obs.n_bl).sum(0)      # noqa: E731
        sums[0] += re(R, R)
        for k in range(4):
            sums[1 + k] -= 2 * re(R, V[1 + k])
        for k, (p, q) in enumerate(((1, 1), (1, 2), (2, 2), (3, 3), (3, 4), (4, 4), (1, 3), (1, 4), (2, 3), (2, 4))):
            sums[5 + k] += 2 * re(V[p], V[q])
    g = torch.zeros((obs.n_ant, 2), dtype=torch.float64, device=DEV)
    H = torch.zeros((obs.n_ant, 3), dtype=torch.float64, device=DEV)
    g.index_add_(0, obs.i, sums[1:3].T).index_add_(0, obs.j, sums[3:5].T)
    H.index_add_(0, obs.i, sums[5:8].T).index_add_(0, obs.j, sums[8:11].T)
    return [float(sums[0].sum()), g.cpu().numpy(), H.cpu().numpy(), np.ascontiguousarray(sums[11:].T.cpu().numpy())]


def _step(obs, ev, lam):
    """The step of the damped system (H + lam diag H) delta = -g."""
    n = obs.n_ant
    A = np.zeros((n, 2, n, 2))
    k = np.arange(n)
    A[k, 0, k, 0], A[k, 0, k, 1], A[k, 1, k, 0], A[k, 1, k, 1] = ev[2][:, 0], ev[2][:, 1], ev[2][:, 1], ev[2][:, 2]
    i, j, x = obs.i.cpu().numpy(), obs.j.cpu().numpy(), ev[3].reshape(-1, 2, 2)
    A[i, :, j, :] = x
    A[j, :, i, :] = x.transpose(0, 2, 1)
    A = A.reshape(2 * n, 2 * n)
    A[np.arange(2 * n), np.arange(2 * n)] *= 1.0 + lam
    return np.linalg.solve(A, -ev[1].reshape(-1)).reshape(n, 2)


def _minimise(obs, grid, evals):
    """Offsets and chi^2 that a solve from zero has accepted after so many evaluations (every trial lowers chi^2 until the minimum)."""
    lm, lam = np.zeros((obs.n_ant, 2)), 1e-3
    best = _evaluate(obs, grid, lm)
    for _ in range(evals - 1):
        trial = lm + _step(obs, best, lam)
        ev = _evaluate(obs, grid, trial)
        if not ev[0] < best[0]:
            break
        lm, best, lam = trial, ev, lam / 10
    return lm, best[0]


def _forward(params, x):
    p = torch.from_numpy(params.astype(np.float64)).to(DEV)
    a = (x.double() - p[-104:-52]) / p[-52:]
    zs, acts, ws, o = [], [a], [], 0
    for k, (n_in, n_out) in enumerate(((52, 256), (256, 256), (256, 256), (256, 2))):
        W, b = p[o:o + n_in * n_out].reshape(n_in, n_out), p[o + n_in * n_out:o + (n_in + 1) * n_out]
        o += (n_in + 1) * n_out
        z = acts[-1] @ W + b
        zs.append(z)
        ws.append(W)
        acts.append(z if k == 3 else 0.5 * z * (1 + torch.erf(z / math.sqrt(2))))
    return zs, acts, ws


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        obs, grids = _batch_inputs(case, seed)
        got = [_minimise(o, g, 2) for o, g in zip(obs, grids)]
        return [lm / ARCSEC for lm, _ in got] + [np.array([x for _, x in got])]
    if kind in ("solve", "eval", "predict"):
        obs = _one_input(case, seed)
        grid = obs.sky.grid()
        if kind == "solve":
            lm, chi2 = _minimise(obs, grid, 12)
            return [lm / ARCSEC, np.array(chi2)]
        how = dict(ap=case["ap"], bf16=case["bf16"], exact=case.get("model") == "exact")
        if case.get("model") == "stack":
            how["stack"] = _stack(case, obs)
        lm = _half(obs.lm_true)
        if kind == "eval":
            return [np.asarray(v) for v in _evaluate(obs, grid, lm, **how)]
        V = torch.empty((5, obs.nt, obs.n_bl, obs.nc), dtype=torch.complex128, device=DEV)
        for c in range(obs.nc):
            V[..., c] = _model(obs, c, grid, lm, **dict(how)).reshape(5, obs.nt, obs.n_bl)
        return [V[0], V[1:]] if case["deriv"] else [V[0]]
    if kind == "learned":
        sky, obs = _learned_inputs(case, seed)
        grid, rows = sky.grid(), []
        for o in obs:
            o.uvw, o.vis = o.uvw[::case["stride"]], o.vis[::case["stride"]]
            o.nt = o.uvw.shape[0]
            X, Y = (torch.zeros((25, o.n_bl), dtype=torch.float64, device=DEV) for _ in range(2))
            N = torch.zeros((5, o.n_bl), dtype=torch.float64, device=DEV)
            s = torch.arange(-2.0, 3.0, dtype=torch.float64, device=DEV) * SIGMA_PRIOR
            for c in range(o.nc):
                T, Tu, Tv, _, _ = _degrid(o, c, grid, slice(None), stencil=True)
                a2 = (ALPHA * o.diam * o.freq[c] / C_LIGHT) ** 2
                D = torch.exp(-0.5 * a2 * (s[:, None] ** 2 + s[None] ** 2))
                V = (D[..., None] * T).reshape(25, o.nt, o.n_bl)
                vo = o.vis[..., c].to(torch.complex128)
                re = lambda a, b: o.w_scale * (a.conj() * b).real.sum(-2)        # noqa: E731
                X += re(vo, V)
                Y += re(V, V)
                dl, dm, R = (v.reshape(o.nt, o.n_bl) for v in (1j * math.pi * Tu, 1j * math.pi * Tv, vo.reshape(-1) - T[2, 2]))
                N += torch.stack([-2 * re(R, dl), -2 * re(R, dm), 2 * re(dl, dl), 2 * re(dl, dm), 2 * re(dm, dm)])
            per = torch.cat([X, Y, N]).T
            per = torch.zeros((o.n_ant, 55), dtype=torch.float64, device=DEV).index_add_(0, o.i, per).index_add_(0, o.j, per)
            X, Y, N = per[:, :25], per[:, 25:50], per[:, 50:]
            det = N[:, 2] * N[:, 4] - N[:, 3] ** 2
            newton = torch.stack([-(N[:, 4] * N[:, 0] - N[:, 3] * N[:, 1]) / det, -(N[:, 2] * N[:, 1] - N[:, 3] * N[:, 0]) / det], 1) / SIGMA_PRIOR
            dchi = (-2 * (X - X[:, 12:13]) + Y - Y[:, 12:13]) / Y[:, 12:13]
            rows.append(torch.cat([newton, X / Y, dchi], 1))
        feat = torch.cat(rows)
        return [feat, _forward(_network(seed), feat)[1][-1]]
    if kind == "mlp_grad":
        x, t = _minibatch(case, seed)
        zs, acts, ws = _forward(_network(seed), x)
        err = acts[-1] - t.double()
        d, grads = 2 * err / case["batch"], []
        for k in (3, 2, 1, 0):
            grads = [(acts[k].T @ d).reshape(-1), d.sum(0)] + grads
            if k:
                z = zs[k - 1]
                d = (d @ ws[k].T) * (0.5 * (1 + torch.erf(z / math.sqrt(2))) + z * torch.exp(-z * z / 2) / math.sqrt(2 * math.pi))
        return [err.square().sum() / case["batch"], torch.cat(grads + [torch.zeros(104, dtype=torch.float64, device=DEV)])]
    if kind == "grid":
        n, ng = case["n_img"], case["n_grid"]
        pad = torch.zeros((ng, ng), dtype=torch.float64, device=DEV)
        at = ng // 2 - n // 2
        pad[at:at + n, at:at + n] = _image(case, seed).double()
        return torch.fft.fftshift(torch.fft.ifft2(torch.fft.ifftshift(pad), norm="forward"))
    comp = torch.from_numpy(_components(case, seed)).to(DEV)
    ng = case["n_grid"]
    u = (torch.arange(ng, dtype=torch.float64, device=DEV) - ng // 2) / (ng * case["cell"] * ARCSEC)
    one = torch.ones((), dtype=torch.float64, device=DEV)
    a = torch.polar(one, 2 * math.pi * u[:, None] * comp[None, :, 0]) * comp[None, :, 2]
    return torch.polar(one, 2 * math.pi * u[:, None] * comp[None, :, 1]) @ a.T
