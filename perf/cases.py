"""Performance cases of the photon Monte Carlo library, through its public Python entry points.

Each case is something a user's program does with the library: expose an image of a scene (Scene.trace in its
three precisions), read every photon's record, differentiate star moments with respect to the optics
(Scene.grad, psf_moments), or saturate a finished image (bleed).  prepare() makes what such a program holds
before the call (a loaded scene and its output buffers); run() is one exposure, gradient or pass; exact() is
the same photons in plain torch, in 64 bits, written from the definitions in include/phosim.h.

Scenes come from the recipes in paper_1504_06570_gb300/inputs.py; the phase screens of the large ones are
drawn on the GPU from the same power spectrum, because the recipes' CPU synthesis takes half a minute.
"""
import functools
import math

import numpy as np
import torch

from paper_1504_06570_gb300 import inputs as I
from paper_1504_06570_gb300 import phosim as P

MAX_GHOST_BOUNCES = 8          # PHOSIM_MAX_GHOST_BOUNCES of include/phosim.h
PRECISIONS = {"fp64": P.PLAIN_FP64, "mixed": P.MIXED, "ds": P.MIXED_DS}


def listed():
    return [
        # a postage stamp: one star on a small chip, the call of a PSF fit or of an interactive look
        {"name": "star_small", "kind": "star", "precision": "ds", "photons": 10_000, "screen": 512, "chip": 256,
         "records": False},
        # the plain-method case of the reference measurements: one star in FP64, every photon's record read back
        {"name": "star_records", "kind": "star", "precision": "fp64", "photons": 100_000, "screen": 512, "chip": 256,
         "records": True},
        # a star field through the survey telescope in the fast precision (the 1e8-photon workload)
        {"name": "field_ds", "kind": "field", "precision": "ds", "photons": 100_000_000, "stars": 1000, "screen": 4096,
         "host_image": False, "graph": False},
        # the same kind of field in the two FP64 precisions (validation runs); an odd screen size in one
        {"name": "field_fp64", "kind": "field", "precision": "fp64", "photons": 20_000_000, "stars": 300, "screen": 2048,
         "host_image": False, "graph": False},
        {"name": "field_mixed", "kind": "field", "precision": "mixed", "photons": 15_000_000, "stars": 777, "screen": 1500,
         "host_image": False, "graph": False},
        # a short exposure added to an image that the user's program keeps in pinned host memory
        {"name": "field_host", "kind": "field", "precision": "ds", "photons": 3_000_000, "stars": 100, "screen": 1024,
         "host_image": True, "graph": False},
        # a quarter of the batched survey workload: stars, galaxies and the bundled sky, replayed as a graph
        {"name": "catalogue", "kind": "catalogue", "sources": 10_000, "scale": 0.25, "screen": 4096, "graph": True,
         "bundle": 8},
        # an engineering run with every optional effect: misalignments, mirror figures, ghosts, second kick, fringing
        {"name": "options_ds", "kind": "options", "precision": "ds", "photons": 4_000_000, "stars": 37, "screen": 511},
        # the differentiation workload: an 8 x 8 star grid and all 97 per-surface parameters
        {"name": "gradient", "kind": "gradient", "side": 8, "photons": 30_000, "parameters": "all"},
        # one iteration of an alignment fit: moments and their gradient for a few parameters and few photons
        {"name": "fit", "kind": "fit", "side": 3, "photons": 2_000, "parameters": "alignment"},
        # saturation of a finished full-chip image with bright stars, and of an odd-sized crowded one
        {"name": "bleed_chip", "kind": "bleed", "nx": 4096, "ny": 4096, "stars": 300, "well": 1000},
        {"name": "bleed_odd", "kind": "bleed", "nx": 1023, "ny": 517, "stars": 200, "well": 1000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["star", "field", "field", "field", "catalogue", "options", "gradient", "fit", "bleed", "bleed"])
    if kind == "star":
        precision = rng.choice(["ds", "mixed", "fp64"])
        return {"kind": kind, "precision": precision, "photons": _log(rng, 1_000, 2_000_000),
                "screen": rng.choice([256, 300, 511, 512]), "chip": rng.randrange(65, 513), "records": rng.random() < 0.5}
    if kind == "field":
        precision = rng.choice(["ds", "ds", "mixed", "fp64"])
        host = rng.random() < 0.3
        return {"kind": kind, "precision": precision,
                "photons": _log(rng, 100_000, 100_000_000 if precision == "ds" and not host else 20_000_000),
                "stars": _log(rng, 1, 1500), "screen": rng.choice([513, 1024, 1500, 2048, 4096]), "host_image": host,
                "graph": not host and rng.random() < 0.5}
    if kind == "catalogue":
        return {"kind": kind, "sources": _log(rng, 200, 10_000), "scale": math.exp(rng.uniform(math.log(0.01), math.log(0.2))),
                "screen": rng.choice([1024, 1777, 2048]), "graph": rng.random() < 0.5, "bundle": rng.choice([1, 5, 8])}
    if kind == "options":
        return {"kind": kind, "precision": rng.choice(["ds", "mixed", "fp64"]), "photons": _log(rng, 100_000, 4_000_000),
                "stars": _log(rng, 1, 200), "screen": rng.choice([256, 333, 511])}
    if kind == "gradient":
        return {"kind": kind, "side": rng.randrange(2, 9), "photons": _log(rng, 1_000, 30_000),
                "parameters": rng.choice(["all", "alignment", "figure"])}
    if kind == "fit":
        return {"kind": kind, "side": rng.randrange(2, 6), "photons": _log(rng, 500, 10_000),
                "parameters": rng.choice(["alignment", "figure"])}
    return {"kind": "bleed", "nx": rng.randrange(64, 4097), "ny": rng.randrange(64, 4097), "stars": _log(rng, 20, 400),
            "well": _log(rng, 300, 5_000)}


# ---------------------------------------------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=2)
def _mode_amplitude(n, pixel_m, low_fcut):
    """Square root of the screen's mode power at r0 = 1 m (it scales with r0^(-5/3)), on the GPU."""
    power = I.fft_mode_power(n, pixel_m, 1.0, 20.0, "all" if low_fcut is None else "low", low_fcut)
    return torch.from_numpy(np.sqrt(power)).cuda()


def _screen(n, pixel_m, r0_m, generator, low_fcut=None):
    noise = torch.randn((n, n), dtype=torch.complex128, device="cuda", generator=generator) * math.sqrt(2.0)
    modes = noise * (_mode_amplitude(n, pixel_m, low_fcut) * r0_m ** (-5.0 / 6.0))
    return (torch.fft.ifft2(modes).real * (n * n)).cpu().numpy()


def _layers(seed, n):
    """The seven two-scale layers of inputs.von_karman_layers with an n x n fine screen (pixel 1 cm)."""
    rng = np.random.default_rng(seed)
    generator = torch.Generator(device="cuda").manual_seed(seed)
    weights = I.cn2_weights(rng)
    coarse_n = max(16, n // 4)
    fcut = 1.0 / (2.0 * n * 0.01)
    layers = []
    for height, w in zip(I.LAYER_HEIGHTS_KM, weights):
        r0 = 0.15 * w ** (-3.0 / 5.0)
        speed, angle = 10.0 * math.sqrt(-math.log(1.0 - rng.random())), 2.0 * math.pi * rng.random()
        layers.append(I.Layer(z=I.ATM_Z0_MM + height * 1e6, vx=speed * 1e3 * math.cos(angle),
                              vy=speed * 1e3 * math.sin(angle),
                              scales=[I.ScreenScale(10.0, _screen(n, 0.01, r0, generator)),
                                      I.ScreenScale(160.0 * n / coarse_n, _screen(coarse_n, 0.16 * n / coarse_n, r0,
                                                                                  generator, fcut))]))
    return sorted(layers, key=lambda layer: -layer.z)


@functools.lru_cache(maxsize=1)
def _second_kick():
    return I.high_frequency_kick_table(K=1024)[0]


def _scene(case, seed):
    kind = case["kind"]
    if kind == "star":
        s = I.paraboloid_scene(n_photons=case["photons"], seed=seed, screen_n=case["screen"],
                               screen_pix_mm=20.0 * 512 / case["screen"], screen_seed=seed + 1, chip=case["chip"])
        return s
    if kind == "field":
        s = I.three_mirror_scene(n_stars=case["stars"], n_total=case["photons"], seed=seed, atmosphere=False)
        s.layers, s.atmosphere = _layers(seed, case["screen"]), True
        return s
    if kind == "catalogue":
        # the recipe's own layers are replaced, so they are made as small as it allows
        s = I.batched_scene(n_sources=case["sources"], seed=seed, fine_n=16, coarse_n=16, photon_scale=case["scale"],
                            background_photons=100_000 * case["sources"], sky_bundle=case["bundle"])
        s.layers = _layers(seed, case["screen"])
        return s
    if kind == "options":
        s = I.three_mirror_scene(n_stars=case["stars"], n_total=case["photons"], seed=seed, atmosphere=False)
        rng = np.random.default_rng(seed)
        s.layers, s.atmosphere = _layers(seed, case["screen"]), True
        for k, mirror in enumerate(s.surfaces[:3]):          # 30 nm rms of figure and a slight misalignment
            c = rng.normal(size=19)
            mirror.zern = (0.0, 0.0, 0.0) + tuple(c / np.sqrt(np.sum(c * c)) * 30e-6)
            mirror.zern_rnorm = mirror.r_out
            mirror.pert = tuple(rng.normal(size=3) * 0.02) + tuple(rng.normal(size=3) * 2e-6)
        for lens in s.surfaces[3:7]:
            lens.pert = tuple(rng.normal(size=3) * 0.01) + tuple(rng.normal(size=3) * 1e-5)
        # an antireflection coating in two angle bins on two lens faces; the filter reflects what it does not pass
        lam = 300.0 + np.arange(900) + 0.5
        ar = np.stack([0.98 - 1e-5 * np.abs(lam - 600.0), 0.97 - 1e-5 * np.abs(lam - 600.0)], 1)
        s.coatings[0].reflect = 0.9 * (1.0 - s.coatings[0].table)
        s.coatings.append(I.Coating(lam0=300.0, dlam=1.0, theta0=0.0, dtheta=0.25, table=ar, reflect=1.0 - ar))
        s.surfaces[4].coating = s.surfaces[5].coating = 1
        s.hf_kick = _second_kick()
        s.back_reflect = s.fringe = True
        s.detector.dead_layer, s.detector.t_si_gx, s.detector.t_si_gy = 1e-4, 2e-5, -1e-5
        s.detector.sigma = I.diffusion_sigma_table(n=33)
        return s
    s, _, _ = I.grad_grid_scene(n_side=case["side"], photons=case["photons"], seed=seed)
    return s


def _parameters(case):
    camera = range(3, 12)
    alignment = [(1, f) for f in (0, 1, 3, 4)] + [(c, f) for c in camera for f in (0, 1, 3, 4)]
    figure = [(m, 100 + j) for m in range(3) for j in range(3, 22)]
    if case["parameters"] == "all":
        return alignment + figure
    return alignment[:8] if case["parameters"] == "alignment" else figure[:19]


def _weights(case, seed):
    """The derivative of a fit's loss with respect to the moments: any numbers of order one."""
    return np.random.default_rng(seed + 77).normal(size=(case["side"] ** 2, 5))


def _crowded_image(case, seed):
    """A finished image in electrons: sky, and stars of which the brightest are far above the full well."""
    rng = np.random.default_rng(seed)
    nx, ny = case["nx"], case["ny"]
    image = torch.poisson(torch.full((ny, nx), 60.0, device="cuda"),
                          generator=torch.Generator(device="cuda").manual_seed(seed)).to(torch.int32)
    for _ in range(case["stars"]):
        x, y = rng.uniform(0, nx), rng.uniform(0, ny)
        flux, sigma = 10 ** rng.uniform(4.0, 6.5), rng.uniform(2.0, 3.0)
        x0, y0 = max(0, int(x) - 20), max(0, int(y) - 20)
        x1, y1 = min(nx, int(x) + 21), min(ny, int(y) + 21)
        gx = np.exp(-0.5 * ((np.arange(x0, x1) + 0.5 - x) / sigma) ** 2)
        gy = np.exp(-0.5 * ((np.arange(y0, y1) + 0.5 - y) / sigma) ** 2)
        light = flux / (2.0 * math.pi * sigma * sigma) * gy[:, None] * gx[None, :]
        image[y0:y1, x0:x1] += torch.from_numpy(light.astype(np.int32)).cuda()
    return image


# ---------------------------------------------------------------------------------------------------------------
# the cases' entry points
# ---------------------------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "bleed":
        image = _crowded_image(case, seed)
        return {"case": case, "raw": image, "image": image.clone()}
    s = _scene(case, seed)
    if kind in ("gradient", "fit"):
        scene = P.Scene(s, P.PLAIN_FP64)
        params = _parameters(case)
        if kind == "gradient":
            return {"case": case, "scene": scene, "params": params, "dL": _weights(case, seed)}
        theta = torch.zeros(len(params), dtype=torch.float64)
        for k, (surface, field) in enumerate(params):
            theta[k] = s.surfaces[surface].zern[field - 100] if field >= 100 else 0.0
        return {"case": case, "scene": scene, "params": params, "theta": theta.requires_grad_(),
                "dL": torch.from_numpy(_weights(case, seed))}
    d = s.detector
    scene = P.Scene(s, PRECISIONS[case.get("precision", "ds")], early_reject=kind != "star", graph=case.get("graph", False))
    host = case.get("host_image", False)
    image = torch.zeros((d.ny, d.nx), dtype=torch.int32, device="cpu" if host else "cuda", pin_memory=host)
    moments = torch.zeros((len(s.sources), P.MOMENT_WORDS), dtype=torch.float64, device="cuda")
    records = torch.zeros((case["photons"], P.RECORD_DTYPE.itemsize), dtype=torch.uint8, device="cuda") \
        if case.get("records") else None
    return {"case": case, "scene": scene, "image": image, "moments": moments, "records": records}


def run(state):
    kind = state["case"]["kind"]
    if kind == "bleed":                            # the raw image is kept
        state["image"].copy_(state["raw"])
        return {"image": state["image"], "removed": P.bleed(state["image"], state["case"]["well"])}
    scene = state["scene"]
    if kind == "gradient":
        gradient, moments = scene.grad(state["dL"], state["params"])
        return {"gradient": gradient, "moments": moments}
    if kind == "fit":
        theta = state["theta"]
        theta.grad = None
        moments = P.psf_moments(theta, scene, state["params"])
        moments.backward(state["dL"])
        return {"moments": moments.detach(), "gradient": theta.grad}
    image, moments, records = state["image"], state["moments"], state["records"]
    image.zero_()
    moments.zero_()
    scene.trace(image, records, moments)
    out = {"image": image, "moments": moments}
    if records is not None:
        out["photons"] = records.view(torch.float64)[:, :5]
        out["fates"] = records.view(torch.int32)[:, 10:]
    return out


# Operations of the method, counted as sums, products, quotients and roots of the 64-bit definition: per photon
# that is followed to the end about 690 of sampling and seven layers and 2600 of optics and sensor in the
# three-mirror telescope (a third of that for the two-surface one with one layer); of the field's photons 19 %
# pass the filter's band.  The adjoint is about twice the optics again.
def work(case):
    kind = case["kind"]
    if kind == "bleed":
        pixels = case["nx"] * case["ny"]
        return {"bytes": 8 * pixels, "flops": 0}
    if kind in ("gradient", "fit"):
        photons = case["side"] ** 2 * case["photons"]
        return {"bytes": case["side"] ** 2 * (168 + 40 + 8 * len(_parameters(case))), "flops": 0.19 * photons * 3 * 2600}
    if kind == "star":
        n, chip = case["photons"], case["chip"] ** 2
        return {"bytes": 4 * chip + 32 * n + (48 * n if case["records"] else 0) + 232, "flops": 700.0 * n}
    chip = 4096 * 4096
    screens = 7 * case["screen"] ** 2 * 8
    if kind == "catalogue":
        # counts log-uniform on 1e2-1e7: 8.7e5 on average; the sky's rays carry a bundle of photons each
        stars, sky = 8.7e5 * case["sources"] * case["scale"], 1e5 * case["sources"] * case["scale"]
        rays = 0.19 * (stars + sky / case["bundle"])
        return {"bytes": 4 * chip + min(screens, rays * 7 * 32) + 232 * case["sources"],
                "flops": 3300.0 * rays + 100.0 * 0.19 * sky}
    n = case["photons"]
    return {"bytes": 4 * chip * (2 if case.get("host_image") else 1) + min(screens, 0.19 * n * 7 * 32) + 232 * case["stars"],
            "flops": 3300.0 * 0.19 * n}


# ---------------------------------------------------------------------------------------------------------------
# the same photons in plain torch, in 64 bits
# ---------------------------------------------------------------------------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind == "bleed":                            # whole numbers
        return None
    if kind == "catalogue" and case["sources"] * case["scale"] > 200:    # over 2e8 photons: more than 20 s
        return None
    with torch.device("cuda"):
        s = _scene(case, seed)
        path = _Path(s)
        if kind in ("gradient", "fit"):
            return _exact_gradient(case, seed, s, path)
        moments, rows = path.moments(want_photons=bool(case.get("records")))
        out = {"image": None, "moments": moments}
        if rows is not None:
            out["photons"], out["fates"] = rows, None
        return out


def _exact_gradient(case, seed, s, path):
    params, dL = _parameters(case), torch.from_numpy(_weights(case, seed)).cuda()
    n = len(s.sources)
    theta = torch.zeros((n, len(params)), dtype=torch.float64, requires_grad=True)
    src, x, y, _, _ = path.detected(0, path.total, theta, params)
    count = torch.bincount(src, minlength=n).double()
    per = lambda v: torch.zeros(n, dtype=torch.float64).index_add(0, src, v) / count  # noqa: E731
    mx, my = per(x), per(y)
    dx, dy = x - mx[src], y - my[src]
    moments = torch.stack([mx, my, per(dx * dx), per(dx * dy), per(dy * dy)], 1)
    (gradient,) = torch.autograd.grad((moments * dL).sum(), theta)
    if case["kind"] == "fit":
        return {"moments": moments.detach(), "gradient": gradient.sum(0)}
    return {"gradient": gradient, "moments": torch.cat([count[:, None], moments.detach()], 1)}


def _philox(c, key):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    low = 0xFFFFFFFF
    k0, k1 = key & low, key >> 32
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = ((p1 >> 32 & low) ^ c[1] ^ k0, p1 & low, (p0 >> 32 & low) ^ c[3] ^ k1, p0 & low)
        k0, k1 = k0 + 0x9E3779B9 & low, k1 + 0xBB67AE85 & low
    return c


def _uniform(w):
    return (w.double() + 0.5) * 2.0 ** -32


def _table(t, f):
    """Linear interpolation of a table at fractional index f, clamped."""
    k = f.floor().long().clamp(0, t.shape[-1] - 2)
    w = (f - k).clamp(0.0, 1.0)
    return t[k] * (1.0 - w) + t[k + 1] * w


def _noll(j):
    """Noll index -> (n, m, is the cosine term)."""
    n = 0
    while (n + 1) * (n + 2) // 2 < j:
        n += 1
    k = j - n * (n + 1) // 2 - 1
    m = 2 * ((k + 1) // 2) if n % 2 == 0 else 2 * (k // 2) + 1
    return n, m, j % 2 == 0


@functools.lru_cache(maxsize=None)
def _zernike(j):
    """Z_j of the unit disk as {(power of x, power of y): coefficient}."""
    n, m, cosine = _noll(j)
    radial = np.poly1d([0.0])
    for k in range((n - m) // 2 + 1):       # in t = x^2 + y^2, divided by rho^m
        c = (-1) ** k * math.factorial(n - k) / (math.factorial(k) * math.factorial((n + m) // 2 - k)
                                                 * math.factorial((n - m) // 2 - k))
        radial = radial + c * np.poly1d([1.0] + [0.0] * ((n - m) // 2 - k))
    norm = math.sqrt(n + 1.0) * (math.sqrt(2.0) if m else 1.0)
    out = {}
    for q, c in enumerate(radial.coeffs[::-1]):
        for a in range(q + 1):
            for b in range(m + 1):          # (x + i y)^m
                i = 1j ** b
                part = (i.real if cosine or m == 0 else i.imag) * math.comb(m, b)
                if part and c:
                    power = (2 * a + m - b, 2 * (q - a) + b)
                    out[power] = out.get(power, 0.0) + norm * c * math.comb(q, a) * part
    return out


_POWERS = [(a, b) for b in range(7) for a in range(7 - b)]


@functools.lru_cache(maxsize=1)
def _zernike_matrix():
    return torch.tensor([[_zernike(j).get(p, 0.0) for p in _POWERS] for j in range(1, 29)], dtype=torch.float64)


def _sellmeier(m, lam):
    l2 = (lam * 1e-3) ** 2
    return torch.sqrt(1.0 + sum(b * l2 / (l2 - c) for b, c in zip(m.B, m.C)))


def _silicon(lam):
    e = 1239.841984 / lam
    return 3.36 + 0.211 * e + 2.79 * torch.exp((e - 3.30) / 0.398)


def _film(lam, n0, n1, k1, t, c1):
    """Reflectance of one silicon layer between a medium of index n0 and vacuum, mean of both polarisations."""
    cpx = lambda v: v.to(torch.complex128)  # noqa: E731
    s2 = n1 ** 2 * (1.0 - c1 ** 2).clamp(min=0.0)
    q0, q2 = torch.sqrt(cpx(n0 ** 2 - s2)), torch.sqrt(cpx(1.0 - s2))
    N1 = torch.complex(n1, k1) ** 2
    q1 = torch.sqrt(N1 - s2)
    e = torch.exp(4j * math.pi * t / (lam * 1e-6) * q1)
    out = 0.0
    for r01, r12 in (((q0 - q1) / (q0 + q1), (q1 - q2) / (q1 + q2)),
                     ((N1 * q0 - n0 ** 2 * q1) / (N1 * q0 + n0 ** 2 * q1), (q1 - N1 * q2) / (q1 + N1 * q2))):
        out = out + 0.5 * ((r01 + r12 * e) / (1.0 + r01 * r12 * e)).abs() ** 2
    return out


class _Path:
    """The photon path of a scene, many photons at a time."""

    def __init__(self, s):
        self.s, src = s, s.sources
        f8 = lambda v: torch.as_tensor(np.array(v, np.float64)).cuda()  # noqa: E731
        self.f8 = f8
        self.col = {k: f8(getattr(src, k)) for k in ("xi", "eta", "redshift", "t0", "t_exp", "a", "b", "pa")}
        self.kind, self.sed, self.sersic_row = (torch.as_tensor(np.asarray(getattr(src, k), np.int64)).cuda()
                                                for k in ("kind", "sed", "table"))
        n = len(src)
        self.bundle = torch.as_tensor(np.ones(n, np.int64) if src.bundle is None else
                                      np.maximum(1, src.bundle).astype(np.int64)).cuda()
        self.spread = f8(np.zeros(n) if src.bundle_sigma is None else src.bundle_sigma)
        self.ends = torch.as_tensor(np.cumsum(src.n_photons.astype(np.int64))).cuda()
        self.total = int(self.ends[-1])
        weight = f8(s.sed_flux) * (s.sed_lam0 + (torch.arange(s.sed_flux.shape[1]) + 0.5) * s.sed_dlam) * s.sed_dlam
        cdf = torch.cumsum(weight, 1)
        self.cdf = cdf / cdf[:, -1:]
        self.screens = [[(sc.pixel, self._nodes(f8(sc.phase), sc.pixel)) for sc in layer.scales] for layer in s.layers]
        self.sersic, self.ell, self.sigma = f8(s.sersic), f8(s.detector.ell), f8(s.detector.sigma)
        self.hf = None if s.hf_kick is None else f8(s.hf_kick)
        self.coat = [(f8(c.table), None if c.reflect is None else f8(np.broadcast_to(c.reflect, c.table.shape)))
                     for c in s.coatings]
        self.slots = [k for k, surf in enumerate(s.surfaces) if surf.coating >= 0 and surf.kind != I.DETECTOR]

    @staticmethod
    def _nodes(ph, pixel):
        gx = (torch.roll(ph, -1, 1) - torch.roll(ph, 1, 1)) / (2.0 * pixel)
        gy = (torch.roll(ph, -1, 0) - torch.roll(ph, 1, 0)) / (2.0 * pixel)
        return torch.stack([gx, gy], -1)

    def words(self, src, ray, block):
        b = torch.as_tensor(block).expand_as(ray)
        return _philox((ray & 0xFFFFFFFF, ray >> 32, src, b), self.s.seed)

    # -- sampling and atmosphere --------------------------------------------------------------------------------
    def entry(self, src, ray):
        """Wavelengths and the words of the first block."""
        s, col = self.s, {k: v[src] for k, v in self.col.items()}
        w0 = self.words(src, ray, 0)
        # the bin of the wavelength draw: the first whose cumulative probability exceeds it
        u, bins = _uniform(w0[2]), torch.empty_like(src)
        for q in torch.unique(self.sed[src]).tolist():
            at = self.sed[src] == q
            bins[at] = torch.searchsorted(self.cdf[q], u[at], right=True).clamp(max=self.cdf.shape[1] - 1)
        lam = (_uniform(w0[3]) * s.sed_dlam + s.sed_lam0 + bins * s.sed_dlam) * (1.0 + col["redshift"])
        return lam, w0

    def first_coating_passes(self, src, ray, lam):
        """False for photons that the first coated surface can neither transmit nor reflect at any angle."""
        if not self.slots:
            return torch.ones_like(lam, dtype=torch.bool)
        c = self.s.coatings[self.s.surfaces[self.slots[0]].coating]
        T, R = self.coat[self.s.surfaces[self.slots[0]].coating]
        most = (T if R is None else T + R).max(1).values
        il = ((lam - c.lam0) / c.dlam).floor().long().clamp(0, most.shape[0] - 1)
        return _uniform(self.words(src, ray, 2)[2]) < most[il]

    def atmosphere(self, src, ray, lam, w0):
        s, col = self.s, {k: v[src] for k, v in self.col.items()}
        w1 = self.words(src, ray, 1)
        t = col["t0"] + col["t_exp"] * _uniform(w1[0])
        nx, ny = col["xi"], col["eta"]
        u1, ang = _uniform(w1[1]), 2.0 * math.pi * _uniform(w1[2])
        K = self.sersic.shape[1]
        f = u1 * K - 0.5
        k = f.floor().long().clamp(0, K - 2)
        w = (f - k).clamp(0.0, 1.0)
        row = self.sersic_row[src]
        r = self.sersic[row, k] * (1.0 - w) + self.sersic[row, k + 1] * w
        dx, dy = col["a"] * r * torch.cos(ang), col["b"] * r * torch.sin(ang)
        cp, sp = torch.cos(col["pa"]), torch.sin(col["pa"])
        g = col["a"] * torch.sqrt(-2.0 * torch.log(u1))
        kind = self.kind[src]
        nx = nx + torch.where(kind == I.SERSIC, dx * cp - dy * sp, torch.where(kind == I.GAUSS, g * torch.cos(ang), 0.0))
        ny = ny + torch.where(kind == I.SERSIC, dx * sp + dy * cp, torch.where(kind == I.GAUSS, g * torch.sin(ang), 0.0))
        r = torch.sqrt(_uniform(w0[0]) * (s.pupil_r_out ** 2 - s.pupil_r_in ** 2) + s.pupil_r_in ** 2)
        ang = 2.0 * math.pi * _uniform(w0[1])
        x, y = r * torch.cos(ang), r * torch.sin(ang)
        first = s.surfaces[0]
        z = first.z + self.sag(first, x, y)[0]
        rinv = 1.0 / torch.sqrt(1.0 - nx * nx - ny * ny)
        x, y, z = x - nx * rinv * (s.h_top - z), y - ny * rinv * (s.h_top - z), s.h_top
        if s.atmosphere:
            scale = (lam / s.lambda_ref) ** -0.2
            kick = s.lambda_ref * 1e-6 / (2.0 * math.pi) * scale
            for layer, scales in zip(s.layers, self.screens):
                x, y, z = x + nx * rinv * (z - layer.z), y + ny * rinv * (z - layer.z), layer.z
                total = 0.0
                for pixel, nodes in scales:
                    n = nodes.shape[0]
                    fx, fy = (x - layer.vx * t) / pixel, (y - layer.vy * t) / pixel
                    i, j = fx.floor(), fy.floor()
                    tx, ty = (fx - i)[:, None], (fy - j)[:, None]
                    i, j = i.long() % n, j.long() % n
                    i1, j1 = (i + 1) % n, (j + 1) % n
                    grad = (nodes[j, i] * (1 - tx) * (1 - ty) + nodes[j, i1] * tx * (1 - ty)
                            + nodes[j1, i] * (1 - tx) * ty + nodes[j1, i1] * tx * ty)
                    total = total + grad
                nx, ny = nx + kick * total[:, 0], ny + kick * total[:, 1]
                rinv = 1.0 / torch.sqrt(1.0 - nx * nx - ny * ny)
            if self.hf is not None:
                w4 = self.words(src, ray, 4)
                K = self.hf.shape[0]
                a, psi = _table(self.hf, _uniform(w4[0]) * K - 0.5) * scale, 2.0 * math.pi * _uniform(w4[1])
                nx, ny = nx + a * torch.cos(psi), ny + a * torch.sin(psi)
                rinv = 1.0 / torch.sqrt(1.0 - nx * nx - ny * ny)
        nz = -torch.sqrt(1.0 - nx * nx - ny * ny)
        x, y = x + nx * rinv * (z - s.z_entrance), y + ny * rinv * (z - s.z_entrance)
        return torch.stack([x, y, torch.full_like(x, s.z_entrance)], 1), torch.stack([nx, ny, nz], 1)

    # -- optics -------------------------------------------------------------------------------------------------
    @staticmethod
    def sag(surf, x, y, figure=None):
        """Sag and slopes; figure: the photons' monomial coefficients of the Zernike figure."""
        r2 = x * x + y * y
        z, g = torch.zeros_like(x), torch.zeros_like(x)
        if surf.R != 0.0:
            root = torch.sqrt(1.0 - (1.0 + surf.kappa) / surf.R ** 2 * r2)
            z, g = r2 / (surf.R * (1.0 + root)), 1.0 / (surf.R * root)
        for k, a in enumerate(surf.alpha):
            if a != 0.0:
                z, g = z + a * r2 ** ((k + 3) / 2.0), g + (k + 3) * a * r2 ** ((k + 1) / 2.0)
        zx, zy = x * g, y * g
        if figure is not None:
            q = 1.0 / surf.zern_rnorm
            pu, pv = [torch.ones_like(x)], [torch.ones_like(x)]
            for _ in range(6):
                pu.append(pu[-1] * x * q)
                pv.append(pv[-1] * y * q)
            for k, (a, b) in enumerate(_POWERS):
                c = figure[..., k]
                z = z + c * pu[a] * pv[b]
                if a:
                    zx = zx + c * a * q * pu[a - 1] * pv[b]
                if b:
                    zy = zy + c * b * q * pu[a] * pv[b - 1]
        return z, zx, zy

    def chief(self):
        """Where each source's chief ray meets the detector surface (no apertures, no coatings)."""
        s, n = self.s, len(self.s.sources)
        src = torch.arange(n)
        nx, ny = self.col["xi"], self.col["eta"]
        nz = -torch.sqrt(1.0 - nx * nx - ny * ny)
        step = (s.z_entrance - s.surfaces[0].z) / -nz
        X = torch.stack([-nx * step, -ny * step, torch.full_like(nx, s.z_entrance)], 1)
        lam = torch.full_like(nx, s.lambda_ref)
        hit = self.optics(src, src, src, lam, X, torch.stack([nx, ny, nz], 1), bare=True)
        x, y = torch.zeros_like(nx), torch.zeros_like(nx)
        x[hit[0]], y[hit[0]] = hit[1], hit[2]
        return x, y

    def optics(self, src, ray, photon, lam, X, D, theta=None, params=(), bare=False):
        """(index, x, y, xc, yc) of the photons that are detected (bare: that reach the detector surface)."""
        s, last = self.s, len(self.s.surfaces) - 1
        n = len(lam)
        where = {}                                # (surface, field) -> column of theta
        for k, p in enumerate(params):
            where[p] = k
        alive = torch.arange(n)                   # photons under way, with their states
        si, way = torch.zeros(n, dtype=torch.long), torch.ones(n, dtype=torch.long)
        bounces, ghost = torch.zeros(n, dtype=torch.long), torch.zeros(n, dtype=torch.long)
        index = torch.ones(n, dtype=torch.float64)
        before, medium = [], -1
        for surf in s.surfaces:
            before.append(medium)
            medium = medium if surf.kind == I.MIRROR else surf.material
        done = []
        state = (alive, X, D, si, way, bounces, ghost, index)
        while len(state[0]):
            kept = []
            for k in torch.unique(state[3]).tolist():
                if not 0 <= k <= last:            # left the telescope
                    continue
                at = state[3] == k
                # all photons are at one surface unless ghosts are under way
                group = state if bool(at.all()) else tuple(v[at] for v in state)
                new = self._surface(k, src, ray, photon, lam, group, before[k], theta, where, bare)
                if k == last:
                    done.append(new)
                else:
                    kept.append(new)
            if not kept:
                break
            state = kept[0] if len(kept) == 1 else tuple(torch.cat(v) for v in zip(*kept))
        if not done:
            e = torch.zeros(0, dtype=torch.float64)
            return torch.zeros(0, dtype=torch.long), e, e, e, e
        return done[0] if len(done) == 1 else tuple(torch.cat(v) for v in zip(*done))

    def _surface(self, k, src, ray, photon, lam, group, before, theta, where, bare):
        s, surf = self.s, self.s.surfaces[k]
        i, X, D, si, way, bounces, ghost, index = group
        pert = []
        for f in range(6):
            v = torch.full_like(index, float(surf.pert[f]))
            pert.append(v + theta[src[i], where[k, f]] if theta is not None and (k, f) in where else v)
        cx, sx, cy, sy, cz, sz = (fn(pert[3 + q]) for q in range(3) for fn in (torch.cos, torch.sin))
        M = torch.stack([torch.stack([cz * cy, sz * cy, -sy], 1),
                         torch.stack([cz * sy * sx - sz * cx, sz * sy * sx + cz * cx, cy * sx], 1),
                         torch.stack([cz * sy * cx + sz * sx, sz * sy * cx - cz * sx, cy * cx], 1)], 1)
        o = torch.stack([pert[0], pert[1], surf.z + pert[2]], 1)
        p, d = (M @ (X - o)[:, :, None])[:, :, 0], (M @ D[:, :, None])[:, :, 0]
        figure = None
        coef = self.f8(list(surf.zern) + [0.0] * (28 - len(surf.zern)))
        mine = [j for j in range(28) if (k, 100 + j) in where] if theta is not None else []
        if surf.zern_rnorm > 0.0 and (mine or bool((coef != 0.0).any())):
            figure = (coef @ _zernike_matrix())[None]
            if mine:
                more = theta[:, [where[k, 100 + j] for j in mine]] @ _zernike_matrix()[mine]
                figure = figure + more[src[i]]
        # the vertex-side root of the conic, then Newton's method for the other terms
        with torch.no_grad():
            P0, d0 = p.detach(), d.detach()
            fig0 = None if figure is None else figure.detach()
            c = 0.0 if surf.R == 0.0 else 1.0 / surf.R
            kc = (1.0 + surf.kappa) * c
            A = c * (d0[:, 0] ** 2 + d0[:, 1] ** 2) + kc * d0[:, 2] ** 2
            B = c * (P0[:, 0] * d0[:, 0] + P0[:, 1] * d0[:, 1]) + kc * P0[:, 2] * d0[:, 2] - d0[:, 2]
            C = c * (P0[:, 0] ** 2 + P0[:, 1] ** 2) + kc * P0[:, 2] ** 2 - 2.0 * P0[:, 2]
            q = -(B + torch.copysign(torch.sqrt(B * B - A * C), B))
            l = C / q
            l = torch.where((A != 0.0) & (1.0 - kc * (P0[:, 2] + l * d0[:, 2]) < 0.0), q / A, l)
            for _ in range(8):
                h = P0 + l[:, None] * d0
                z, zx, zy = self.sag(surf, h[:, 0], h[:, 1], fig0)
                l = l - (h[:, 2] - z) / (d0[:, 2] - zx * d0[:, 0] - zy * d0[:, 1])
            h = P0 + l[:, None] * d0
            _, zx, zy = self.sag(surf, h[:, 0], h[:, 1], fig0)
            slope = d0[:, 2] - zx * d0[:, 0] - zy * d0[:, 1]
        if theta is not None:                     # one more step gives the root its derivative
            h = p + l[:, None] * d
            l = l - (h[:, 2] - self.sag(surf, h[:, 0], h[:, 1], figure)[0]) / slope
        p = p + l[:, None] * d
        _, zx, zy = self.sag(surf, p[:, 0], p[:, 1], figure)
        N = torch.stack([-zx, -zy, torch.ones_like(zx)], 1) / torch.sqrt(1.0 + zx * zx + zy * zy)[:, None]
        ok = torch.isfinite(l.detach()) & ((bounces == 0) | (l.detach() > 0.0))

        def refract(d, N, mu):
            cosi = -(d * N).sum(1)
            N, cosi = torch.where(cosi < 0.0, -1.0, 1.0)[:, None] * N, cosi.abs()
            k = 1.0 - mu * mu * (1.0 - cosi * cosi)
            return mu[:, None] * d + (mu * cosi - torch.sqrt(k.clamp(min=0.0)))[:, None] * N, k >= 0.0

        if surf.kind == I.DETECTOR:
            return self._sensor(src, ray, photon, lam, i, p, d, N, index, ok, refract, bare)
        turned = torch.zeros_like(ok)
        if not bare:
            r2 = (p[:, :2].detach() ** 2).sum(1)
            ok &= (r2 <= surf.r_out ** 2) & (r2 >= surf.r_in ** 2)
            if k in self.slots:
                c, (T, R) = s.coatings[surf.coating], self.coat[surf.coating]
                th = torch.arccos((d * N).detach().sum(1).abs().clamp(max=1.0))
                it = ((th - c.theta0) / c.dtheta).floor().long().clamp(0, T.shape[1] - 1)
                il = ((lam[i] - c.lam0) / c.dlam).floor().long().clamp(0, T.shape[0] - 1)
                slot = self.slots.index(k)
                w = self.words(src[i], ray[i], 2 if slot < 2 else 3)[2 + slot if slot < 2 else slot - 2]
                if bool((bounces > 0).any()):
                    g = torch.stack(self.words(src[i], ray[i], 7 + ghost // 4), 1).gather(1, (ghost % 4)[:, None])[:, 0]
                    w = torch.where(bounces > 0, g, w)
                    ghost = ghost + (bounces > 0)
                u, T0 = _uniform(w), T[il, it]
                passed = u < T0
                if R is not None and surf.kind == I.REFRACT:
                    turned = ~passed & (u < T0 + R[il, it])
                    bounces = bounces + turned
                    turned &= bounces <= MAX_GHOST_BOUNCES
                ok &= passed | turned
        mirrored = d - 2.0 * (d * N).sum(1)[:, None] * N
        if surf.kind == I.MIRROR:
            d = mirrored
        else:
            after = torch.empty_like(index)
            for material, at in ((surf.material, way > 0), (before, way < 0)):
                m = s.materials[material] if material >= 0 else I.Material()
                n = _sellmeier(m, lam[i]) if m.kind == I.SELLMEIER else _silicon(lam[i]) if m.kind == I.SILICON \
                    else torch.ones_like(index)
                after = torch.where(at, n, after)
            through, fine = refract(d, N, index / after)
            ok &= fine | turned
            d = torch.where(turned[:, None], mirrored, through)
            index = torch.where(turned, index, after)
            way = torch.where(turned, -way, way)
        X, D = (p[:, None, :] @ M)[:, 0] + o, (d[:, None, :] @ M)[:, 0]
        group = (i, X, D, si + way, way, bounces, ghost, index)
        return group if bool(ok.all()) else tuple(v[ok] for v in group)

    def _sensor(self, src, ray, photon, lam, i, p, d, N, index, ok, refract, bare):
        s, det = self.s, self.s.detector
        if bare:
            return tuple(v[ok] for v in (i, p[:, 0], p[:, 1], p[:, 0], p[:, 1]))
        xlo, ylo = det.x0 - 0.5 * det.nx * det.pixel, det.y0 - 0.5 * det.ny * det.pixel

        def on_chip(x, y):
            fx, fy = torch.floor((x.detach() - xlo) / det.pixel), torch.floor((y.detach() - ylo) / det.pixel)
            return (fx >= 0) & (fy >= 0) & (fx < det.nx) & (fy < det.ny)

        x, y = p[:, 0], p[:, 1]
        w1, w2 = self.words(src[i], ray[i], 1), self.words(src[i], ray[i], 2)
        u = [_uniform(w) for w in (w1[3], w2[0], w2[1], self.words(src[i], ray[i], 4)[2])]
        bundled = self.bundle[src[i]] > 1
        if bool(bundled.any()):                   # a photon of a bundle: its offset from the ray's hit, its own draws
            m5, m6 = self.words(src[i], photon[i], 5), self.words(src[i], photon[i], 6)
            g = self.spread[src[i]] * torch.sqrt(-2.0 * torch.log(_uniform(m5[0])))
            psi = 2.0 * math.pi * _uniform(m5[1])
            x = x + torch.where(bundled, g * torch.cos(psi), 0.0)
            y = y + torch.where(bundled, g * torch.sin(psi), 0.0)
            u = [torch.where(bundled, _uniform(m), v) for m, v in zip((m5[2], m5[3], m6[0], m6[1]), u)]
        ok &= on_chip(x, y)
        xc, yc = x, y
        on, lost_row = ok, torch.stack([torch.zeros_like(x), torch.zeros_like(x), x, y], 1)
        if s.sensor:
            lam = lam[i]
            n_si = _silicon(lam)
            d, fine = refract(d, N, index / n_si)
            ok = ok & fine
            ell = _table(self.ell, (lam - det.ell_lam0) / det.ell_dlam)
            L = -ell * torch.log(u[0])
            depth = L * d[:, 2].detach().abs()
            through = depth > det.t_si
            if s.back_reflect:
                if s.fringe:
                    t = det.t_si + det.t_si_gx * (x - det.x0) + det.t_si_gy * (y - det.y0)
                    back = _film(lam, index, n_si, lam * 1e-6 / (4.0 * math.pi * ell), t, d[:, 2].abs())
                else:
                    back = ((n_si - 1.0) / (n_si + 1.0)) ** 2
                depth = torch.where(through & (u[3] < back),
                                    2.0 * det.t_si - depth, depth)
            ok = ok & (depth >= 0.0) & (depth <= det.t_si) & (depth >= det.dead_layer)
            xc, yc = x + L * d[:, 0], y + L * d[:, 1]
            g = _table(self.sigma, depth * (len(self.sigma) - 1) / det.t_si) * torch.sqrt(-2.0 * torch.log(u[1]))
            psi = 2.0 * math.pi * u[2]
            x, y = xc + g * torch.cos(psi), yc + g * torch.sin(psi)
        # records: a photon lost in the silicon keeps its hit alone
        self.rows = i[on], torch.where(ok[:, None], torch.stack([x, y, xc, yc], 1), lost_row)[on].detach()
        ok = ok & on_chip(x, y)
        return tuple(v[ok] for v in (i, x, y, xc, yc))

    # -- whole calls --------------------------------------------------------------------------------------------
    def detected(self, first, end, theta=None, params=()):
        """(source, x, y) of the detected photons among photons first .. end of the scene, the record rows of those
        that met the detector (their index, x, y, xc, yc) and every photon's wavelength."""
        n = torch.arange(first, end)
        src = torch.searchsorted(self.ends, n, right=True)
        photon = n - torch.where(src > 0, self.ends[(src - 1).clamp(min=0)], 0)
        ray = photon // self.bundle[src]
        lam, w0 = self.entry(src, ray)
        go = self.first_coating_passes(src, ray, lam)
        at, lam_all, w0 = n[go] - first, lam, tuple(w[go] for w in w0)
        src, ray, photon, lam = src[go], ray[go], photon[go], lam[go]
        X, D = self.atmosphere(src, ray, lam, w0)
        self.rows = n[:0], torch.zeros((0, 4), dtype=torch.float64)
        i, x, y, _, _ = self.optics(src, ray, photon, lam, X, D, theta, params)
        return src[i], x, y, (at[self.rows[0]], self.rows[1]), lam_all

    def moments(self, want_photons):
        n = len(self.s.sources)
        rx, ry = self.chief()
        out = torch.zeros((n, 8), dtype=torch.float64)
        out[:, 6], out[:, 7] = rx, ry
        rows = torch.full((self.total, 5), float("nan"), dtype=torch.float64) if want_photons else None
        for first in range(0, self.total, 4_000_000):
            end = min(self.total, first + 4_000_000)
            src, x, y, (at, xy), lam = self.detected(first, end)
            dx, dy = x - rx[src], y - ry[src]
            for k, v in enumerate((torch.ones_like(dx), dx, dy, dx * dx, dx * dy, dy * dy)):
                out[:, k].index_add_(0, src, v)
            if rows is not None:
                rows[first:end] = 0.0
                rows[first + at, :4] = xy
                rows[first:end, 4] = lam
        return out, rows

