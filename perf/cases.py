"""Performance cases of the chi^2 forward-modelling path.

A case is one call of the public Python API on one kind of problem, the way a
fitting program makes it: chi^2 with its gradient (a sampler's or a first-order
optimiser's step), the Levenberg-Marquardt normal equations, a few LM
iterations, or the model images.  The problems are the ones the workloads of
this repository are made of: a single galaxy, batches of independent cutouts,
star and galaxy fields, crowded fields behind a large PSF and a mask, joint
fits of several rotated exposures with shared parameters, overlapping galaxies
without a PSF, and ragged images holding every profile type.

The layout of a problem (image sizes, rotations, positions, sizes of sources,
windows: what the plan is made from) follows from the case, so that results of
two seeds have the same shapes; the light (fluxes, profiles, axis ratios,
angles), the start of the fit, masks and noise come from the seed.  The data
are a float64 model rendered here plus noise of the model's variance.

The mixed form computes in float32 and hands its sums back as float64; its
results are returned as float32, the precision that they carry.  The float64
form's results stay float64.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2308_01957_gb300 import api

# profile codes of the library's source descriptors
SERSIC, EXPONENTIAL, GAUSSIAN, MOFFAT, SKY_FLAT, SKY_PLANE, PSF_STAR = range(7)
SLOTS = {SERSIC: 7, EXPONENTIAL: 6, GAUSSIAN: 6, MOFFAT: 7, SKY_FLAT: 1, SKY_PLANE: 3, PSF_STAR: 3}

STAR_HALF = 16      # half size of a point source's window
LAMBDA0 = 0.1       # damping a fit starts with


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def _case(name, call, layout, height, width, galaxies, stars, psf, **kw):
    c = {"name": name, "call": call, "layout": layout, "height": height, "width": width, "galaxies": galaxies,
         "stars": stars, "psf": psf, "images": 1, "bands": 1, "mask": 0.0, "order": 3, "precision": "mixed",
         "iterations": 0, "live_psf": False}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a sampler or first-order optimiser on one galaxy
        _case("single_eval", "eval", "field", 128, 128, 1, 0, 11),
        # the quick fit of one galaxy on a stamp
        _case("single_lm", "lm", "field", 128, 128, 1, 0, 11, iterations=2),
        # a survey's batch of independent stamps of many sizes, each with its own PSF
        _case("cutouts_lm", "lm", "cutouts", 64, 256, 0, 8, 31, images=64, iterations=2),
        # an ordinary field of galaxies and stars: one gradient, and the first iterations of a fit
        _case("field_eval", "eval", "field", 1024, 1024, 50, 200, 25),
        _case("field_lm", "lm", "field", 1024, 1024, 50, 200, 25, iterations=2),
        # the adaptive pixel integration of the same field, as a check of the fitted model uses it
        _case("field_adaptive", "adaptive", "field", 1024, 1024, 50, 200, 25),
        # a crowded field behind a wide PSF with masked pixels
        _case("crowded_lm", "lm", "field", 1536, 1536, 281, 703, 51, mask=0.02, iterations=2),
        # four exposures in two bands sharing shapes and positions: normal equations for an outside solver
        _case("joint_normal", "normal", "joint", 1024, 1024, 75, 250, 31, images=4, bands=2),
        # the largest: twelve exposures in four bands, a fit's first iterations
        _case("joint_lm", "lm", "joint", 2048, 2048, 300, 1000, 31, images=12, bands=4, iterations=2),
        # large overlapping galaxies without a PSF (the paper's own GPU benchmark)
        _case("overlap_lm", "lm", "overlap", 1000, 1000, 16, 0, 0, iterations=2),
        # model images of ragged, rotated exposures with every profile type, at a higher order
        _case("mixed_render", "render", "mixed", 517, 731, 6, 6, 13, images=3, mask=0.05, order=5),
        # the float64 form, for the reference solution of a small field
        _case("field_f64_normal", "normal", "field", 250, 259, 4, 12, 13, precision="f64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["field", "field", "field", "crowded", "cutouts", "cutouts", "joint", "joint", "overlap", "mixed"])
    call = rng.choice(["eval", "normal", "lm"])
    iterations = rng.randint(1, 2) if call == "lm" else 0   # far from the optimum: clear decisions
    order = rng.choice([1, 3, 3, 3, 3, 5])
    psf = 2 * rng.randint(3, 16) + 1
    common = {"iterations": iterations, "order": order}
    if kind == "field":
        if rng.random() < 0.25:     # the float64 form runs on small fields
            h, w = _log_int(rng, 64, 256), _log_int(rng, 64, 256)
            c = _case("", rng.choice(["eval", "normal"]), "field", h, w, rng.randint(1, 4), rng.randint(0, 12), psf,
                      precision="f64", order=3)
        else:
            h, w = _log_int(rng, 64, 2048), _log_int(rng, 64, 2048)
            area = h * w / 1e6
            call = rng.choice([call, call, call, "render", "adaptive", "shifted"])
            common["iterations"] = iterations if call == "lm" else 0
            c = _case("", call, "field", h, w, max(1, round(48 * area * rng.uniform(0.5, 2.0))),
                      round(190 * area * rng.uniform(0.5, 2.0)), psf, mask=rng.choice([0.0, 0.02]), **common)
    elif kind == "crowded":
        h, w = _log_int(rng, 512, 2048), _log_int(rng, 512, 2048)
        area = h * w / 1e6
        common["order"] = 3
        c = _case("", call, "field", h, w, round(119 * area), round(298 * area), 2 * rng.randint(20, 32) + 1, mask=0.02,
                  **common)
    elif kind == "cutouts":
        lo = rng.randint(32, 96)
        common["order"] = 3
        c = _case("", call, "cutouts", lo, lo + rng.randint(16, 300), 0, rng.randint(2, 8), 31,
                  images=_log_int(rng, 4, 128), **common)
    elif kind == "joint":
        bands, epochs = rng.randint(1, 3), rng.randint(1, 3)
        side = _log_int(rng, 256, 1400)
        common["order"] = 3
        c = _case("", call, "joint", side, side, max(2, round(72 * side * side / 1e6)), round(238 * side * side / 1e6), psf,
                  images=bands * epochs, bands=bands, **common)
    elif kind == "overlap":
        h, w = _log_int(rng, 400, 1200), _log_int(rng, 400, 1200)
        common["order"] = 3
        c = _case("", call, "overlap", h, w, _log_int(rng, 1, 40), 0, 0, **common)
    else:
        live = rng.random() < 0.3
        call = rng.choice(["render", "eval", "normal"] + ([] if live else ["shifted"]))
        c = _case("", call, "mixed", _log_int(rng, 48, 700), _log_int(rng, 48, 900), rng.randint(1, 6),
                  rng.randint(1, 6), 2 * rng.randint(2, 9) + 1, images=rng.randint(1, 3), mask=rng.choice([0.0, 0.05]),
                  order=rng.choice([3, 5, 7]), live_psf=live)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# problems from a seed: numbers only
# ---------------------------------------------------------------------------

def _moffat_rd(fwhm, beta=3.0):
    return fwhm / (2.0 * math.sqrt(2.0 ** (1.0 / beta) - 1.0))


def _psf_image(K, fwhm, wing=False):
    c = (K - 1) / 2.0
    y, x = np.mgrid[0:K, 0:K]
    r2 = (x - c) ** 2 + (y - c) ** 2
    p = (1.0 + r2 / _moffat_rd(fwhm) ** 2) ** -3.0
    p /= p.sum()
    if wing:
        g = np.exp(-r2 / 200.0)
        p += 0.01 * g / g.sum()
    return (p / p.sum()).astype(np.float32)


def _sersic_ie(F, n, Re, q):
    """Surface brightness at Re of a Sersic galaxy of total flux F (b_n by its asymptotic form)."""
    b = 2.0 * n - 1.0 / 3.0 + 4.0 / (405.0 * n)
    return F / (2.0 * math.pi * n * Re * Re * q * math.exp(b - 2.0 * n * math.log(b) + math.lgamma(2.0 * n)))


def _draw_galaxy(lay, rng, xy, re_cap=40.0):
    """A catalogued galaxy: detected well above the sky's noise."""
    n, q, pa = rng.uniform(0.6, 4.5), rng.uniform(0.2, 0.95), rng.uniform(0.0, math.pi)
    Re = min(math.exp(lay.uniform(math.log(2.0), math.log(40.0))), re_cap)
    return [xy[0], xy[1], q, pa, n, Re, _sersic_ie(10.0 ** rng.uniform(3.5, 5.5), n, Re, q)]


def _start_galaxy(rng, p):
    """A fit's starting point near the truth."""
    return [p[0] + rng.normal(0, 0.5), p[1] + rng.normal(0, 0.5), float(np.clip(p[2] * rng.normal(1, 0.1), 0.2, 0.95)),
            p[3] + rng.normal(0, math.radians(5.0)), float(np.clip(p[4] + rng.normal(0, 0.3), 0.5, 6.0)),
            p[5] * rng.normal(1, 0.1), p[6] * rng.normal(1, 0.1)]


class _Problem:
    """Images, sources and parameters; theta is the truth, start where a fit begins."""

    def __init__(self):
        self.images, self.sources, self.theta, self.start = [], [], [], []

    def image(self, H, W, A, origin, psf, group, var_scale=1.0, floor=1.0):
        self.images.append(SimpleNamespace(H=H, W=W, A=A, origin=origin, psf=psf, group=group, var_scale=var_scale,
                                           floor=floor, psf_pidx=None, psf_pfix=None))
        return len(self.images) - 1

    def params(self, true, start):
        base = len(self.theta)
        self.theta.extend(float(v) for v in true)
        self.start.extend(float(v) for v in start)
        return list(range(base, base + len(true)))

    def source(self, kind, image, half, xy, conv, pidx, pfix=None):
        im = self.images[image]
        if half is None:
            win = (0, im.W, 0, im.H)
        else:
            u, v = np.linalg.solve(im.A, np.asarray(xy) - im.origin)
            j, i = math.floor(u), math.floor(v)
            win = (max(j - half, 0), min(j + half + 1, im.W), max(i - half, 0), min(i + half + 1, im.H))
            if win[0] >= win[1] or win[2] >= win[3]:
                return
        idx, fix = np.full(8, -1, dtype=np.int64), np.zeros(8)
        idx[: len(pidx)] = pidx
        for k, v in (pfix or {}).items():
            fix[k] = v
        self.sources.append(SimpleNamespace(type=kind, image=image, win=win, psf_convolve=bool(conv), pidx=idx, pfix=fix))

    def galaxy(self, image, p, idx, conv=True):
        self.source(SERSIC, image, int(min(max(math.ceil(6.0 * p[5]), 16), 256)), p[:2], conv, idx)

    def star(self, image, xy, idx, fwhm=3.0):
        self.source(MOFFAT, image, STAR_HALF, xy, False, [idx[0], idx[1], -1, -1, -1, -1, idx[2]],
                    {2: 1.0, 4: 3.0, 5: _moffat_rd(fwhm)})

    def sky(self, image, plane=True):
        rng_value = [1.0, 1e-4, 1e-4] if plane else [1.0]
        idx = self.params(rng_value, [1.01] + rng_value[1:])
        self.source(SKY_PLANE if plane else SKY_FLAT, image, None, None, False, idx)


def _rotation(phi, scale=1.0):
    return scale * np.array([[math.cos(phi), -math.sin(phi)], [math.sin(phi), math.cos(phi)]])


def _field(c, lay, rng, pr):
    H, W, K = c["height"], c["width"], c["psf"]
    im = pr.image(H, W, np.eye(2), np.zeros(2), _psf_image(K, 3.0, wing=K > 40), 0)
    one = c["galaxies"] == 1 and c["stars"] == 0
    for _ in range(c["galaxies"]):
        xy = lay.uniform([0.4 * W, 0.4 * H], [0.6 * W, 0.6 * H]) if one else lay.uniform([0, 0], [W, H])
        p = _draw_galaxy(lay, rng, xy, max(min(H, W) / 8.0, 2.0))
        pr.galaxy(im, p, pr.params(p, _start_galaxy(rng, p)))
    for _ in range(c["stars"]):
        xy, F = lay.uniform([0, 0], [W, H]), math.exp(rng.uniform(math.log(2e2), math.log(2e4)))
        pr.star(im, xy, pr.params([*xy, F], [*(xy + rng.normal(0, 0.3, 2)), F * rng.normal(1, 0.1)]))
    pr.sky(im, plane=not one)


def _cutouts(c, lay, rng, pr):
    for g in range(c["images"]):
        s = int(lay.integers(c["height"], c["width"] + 1))
        K, fwhm = int(lay.choice(np.arange(15, c["psf"] + 1, 2))), rng.uniform(2.5, 4.0)
        im = pr.image(s, s, np.eye(2), np.zeros(2), _psf_image(K, fwhm), g)
        for _ in range(int(lay.integers(1, c["stars"] + 1))):
            xy = lay.uniform(0.2 * s, 0.8 * s, 2)
            if lay.random() < 0.5:
                p = _draw_galaxy(lay, rng, xy, s / 8.0)
                pr.galaxy(im, p, pr.params(p, _start_galaxy(rng, p)))
            else:
                F = math.exp(rng.uniform(math.log(2e2), math.log(2e4)))
                pr.star(im, xy, pr.params([*xy, F], [*(xy + rng.normal(0, 0.3, 2)), F * rng.normal(1, 0.1)]), fwhm)
        pr.sky(im, plane=False)


def _joint(c, lay, rng, pr):
    side, bands = c["height"], c["bands"]
    per_band = c["images"] // bands
    for i in range(c["images"]):
        A = _rotation(lay.uniform(0, 2 * math.pi))
        origin = lay.uniform(0, 1, 2) - A @ np.full(2, side / 2.0)
        pr.image(side, side, A, origin, _psf_image(c["psf"], rng.uniform(2.5, 4.0)), 0)

    def position():     # in the disc that every rotated image covers
        while True:
            xy = lay.uniform(-0.45 * side, 0.45 * side, 2)
            if xy @ xy < (0.45 * side) ** 2:
                return xy

    for _ in range(c["galaxies"]):
        p = _draw_galaxy(lay, rng, position(), max(side / 8.0, 2.0))
        shape = pr.params(p[:6], _start_galaxy(rng, p)[:6])
        for b in range(bands):
            Ie = p[6] * 10.0 ** rng.normal(0, 0.2)
            idx = pr.params([Ie], [Ie * rng.normal(1, 0.1)])
            for i in range(b * per_band, (b + 1) * per_band):
                pr.galaxy(i, p, shape + idx)
    for _ in range(c["stars"]):
        xy, F = position(), math.exp(rng.uniform(math.log(2e2), math.log(2e4)))
        pos = pr.params(xy, xy + rng.normal(0, 0.3, 2))
        for b in range(bands):
            Fb = F * 10.0 ** rng.normal(0, 0.2)
            idx = pr.params([Fb], [Fb * rng.normal(1, 0.1)])
            for i in range(b * per_band, (b + 1) * per_band):
                pr.star(i, xy, pos + idx)
    for i in range(c["images"]):
        pr.sky(i)


def _overlap(c, lay, rng, pr):
    H, W = c["height"], c["width"]
    im = pr.image(H, W, np.eye(2), np.zeros(2), None, 0, var_scale=0.01)
    for _ in range(c["galaxies"]):
        p = [lay.uniform(0.05 * W, 0.95 * W), lay.uniform(0.05 * H, 0.95 * H), rng.uniform(0.3, 0.9),
             rng.uniform(0, math.pi), rng.uniform(0.5, 4.0), 10.0 ** lay.uniform(1.5, 2.5), 10.0 ** rng.normal(0, 0.5)]
        s = [p[0] + rng.normal(0, 2), p[1] + rng.normal(0, 2), float(np.clip(p[2] * rng.normal(1, 0.1), 0.3, 0.9)),
             p[3] + rng.normal(0, math.radians(5)), float(np.clip(p[4] + rng.normal(0, 0.3), 0.5, 4.0)),
             p[5] * rng.normal(1, 0.1), p[6] * rng.normal(1, 0.1)]
        pr.galaxy(im, p, pr.params(p, s), conv=False)


def _mixed(c, lay, rng, pr):
    H, W = c["height"], c["width"]
    live = None
    for i in range(c["images"]):
        A = _rotation(lay.uniform(0, 2 * math.pi), lay.uniform(0.8, 1.2))
        A[0, 1] += 0.05
        psf = _psf_image(c["psf"], 2.0).astype(np.float64) * (1.0 + 0.3 * rng.random((c["psf"], c["psf"])))
        im = pr.image(H, W, A, lay.uniform(0, 1, 2) - A @ np.array([W / 2.0, H / 2.0]), psf.astype(np.float32), 0, floor=0.5)
        if c["live_psf"]:
            live = live or pr.params([2.8, 1.9], [3.1, 1.75])
            pr.images[im].psf_pidx, pr.images[im].psf_pfix = np.array(live, dtype=np.int64), np.zeros(2)

        def place():
            return A @ (lay.uniform(0.1, 0.9, 2) * np.array([W, H])) + pr.images[im].origin

        def near(p):
            return [p[0] + rng.normal(0, 0.2), p[1] + rng.normal(0, 0.2)] + [v * rng.normal(1, 0.03) for v in p[2:]]

        for _ in range(c["galaxies"]):
            xy, q, pa = place(), rng.uniform(0.4, 0.9), rng.uniform(0, math.pi)
            p = [*xy, q, pa, rng.uniform(0.7, 4.0), rng.uniform(2.0, 6.0), rng.uniform(2.0, 10.0)]
            pr.source(SERSIC, im, 24, xy, True, pr.params(p, near(p)))
            xy = place()
            p = [*xy, q, pa, rng.uniform(2.0, 5.0), rng.uniform(1.0, 5.0)]
            pr.source(EXPONENTIAL, im, 20, xy, True, pr.params(p, near(p)))
            xy = place()
            p = [*xy, q, pa, rng.uniform(1.0, 3.0), rng.uniform(20.0, 80.0)]
            pr.source(GAUSSIAN, im, 12, xy, True, pr.params(p, near(p)))
        for _ in range(c["stars"]):
            xy = place()
            p = [*xy, rng.uniform(0.7, 0.95), rng.uniform(0, math.pi), rng.uniform(2.0, 4.0), rng.uniform(1.0, 2.5),
                 rng.uniform(30.0, 100.0)]
            pr.source(MOFFAT, im, 14, xy, False, pr.params(p, near(p)))
            xy = place()
            p = [*xy, rng.uniform(30.0, 90.0)]
            if c["live_psf"]:
                idx = pr.params(p, near(p))
                pr.source(MOFFAT, im, 10, xy, False, [idx[0], idx[1], -1, -1, live[0], live[1], idx[2]], {2: 1.0})
            else:
                pr.source(PSF_STAR, im, 10, xy, False, pr.params(p, near(p)))
        pr.sky(im, plane=i % 2 == 0)


def _build(c, seed):
    rng, pr = np.random.default_rng([int(seed), 23080195]), _Problem()
    lay = np.random.default_rng([c[k] for k in ("height", "width", "galaxies", "stars", "psf", "images", "bands")])
    layouts = {"field": _field, "cutouts": _cutouts, "joint": _joint, "overlap": _overlap, "mixed": _mixed}
    layouts[c["layout"]](c, lay, rng, pr)
    pr.theta, pr.start = np.asarray(pr.theta), np.asarray(pr.start)
    pr.n_groups = 1 + max(im.group for im in pr.images)
    for im in pr.images:
        im.K = 0 if im.psf is None else im.psf.shape[0]
        im.h = max(im.K - 1, 0) // 2
        im.area = abs(float(np.linalg.det(im.A)))
    for s in pr.sources:
        im = pr.images[s.image]
        s.conv = s.psf_convolve and im.K > 0
        h = im.h if s.conv else 0
        s.box = (max(s.win[2] - h, -h), min(s.win[3] + h, im.H + h), max(s.win[0] - h, -h), min(s.win[1] + h, im.W + h))
        s.sup = (max(s.box[0] - h, 0), min(s.box[1] + h, im.H), max(s.box[2] - h, 0), min(s.box[3] + h, im.W))
        s.free = [k for k in range(SLOTS[s.type]) if s.pidx[k] >= 0]
    return pr


# ---------------------------------------------------------------------------
# the same mathematics in plain float64 torch: it makes the data, and the
# values that results are held against
# ---------------------------------------------------------------------------

def _gammainc(a, x):
    return float(torch.special.gammainc(torch.tensor(a, dtype=torch.float64), torch.tensor(x, dtype=torch.float64)))


def _bn_root(n):
    """b with P(2n, b) = 1/2, by bisection and Newton steps."""
    a = 2.0 * n
    b = max(a - 1.0 / 3.0 + 4.0 / (405.0 * n), 0.05)
    for _ in range(60):
        pdf = math.exp((a - 1.0) * math.log(b) - b - math.lgamma(a))
        step = (_gammainc(a, b) - 0.5) / pdf
        b = max(b - step, 0.2 * b)
        if abs(step) < 1e-15 * b:
            break
    return b


def _bn(n, slope):
    """(b_n, db/dn) of a list of n; the slope by central differences of the root."""
    if not slope:   # enough for data: the asymptotic expansion
        b = [2 * v - 1 / 3 + 4 / (405 * v) + 46 / (25515 * v * v) + 131 / (1148175 * v ** 3) for v in n]
        return b, [0.0] * len(n)
    h = 1e-3
    return ([_bn_root(v) for v in n],
            [(8 * (_bn_root(v + h) - _bn_root(v - h)) - (_bn_root(v + 2 * h) - _bn_root(v - 2 * h))) / (12 * h) for v in n])


def _slot_values(pr, s, theta):
    return [theta[s.pidx[k]] if s.pidx[k] >= 0 else s.pfix[k] for k in range(SLOTS[s.type])]


class _Batch:
    """Sources of one image, one type and one box shape, evaluated together."""

    def __init__(self, pr, sources, theta, order, exact=True):
        s0 = sources[0]
        self.sources, self.kind, self.im = sources, s0.type, pr.images[s0.image]
        self.p = torch.tensor([_slot_values(pr, s, theta) for s in sources], dtype=torch.float64, device="cuda")
        box = torch.tensor([s.box for s in sources], dtype=torch.float64, device="cuda")
        x, w = np.polynomial.legendre.leggauss(order)
        t = [(x[a] / 2, x[b] / 2, w[a] * w[b] / 4) for b in range(order) for a in range(order)]
        self.nodes = [torch.tensor(v, dtype=torch.float64, device="cuda").view(1, -1, 1, 1) for v in zip(*t)]
        h, wd = s0.box[1] - s0.box[0], s0.box[3] - s0.box[2]
        self.i = (box[:, 0, None] + torch.arange(h, dtype=torch.float64, device="cuda") + 0.5)[:, None, :, None]
        self.j = (box[:, 2, None] + torch.arange(wd, dtype=torch.float64, device="cuda") + 0.5)[:, None, None, :]
        if self.kind == SERSIC:
            n = self.p[:, 4].tolist()
            self.b, self.db, self.n0 = (torch.tensor(v, dtype=torch.float64, device="cuda") for v in (*_bn(n, exact), n))

    def values(self, p):
        """Pixel values (N, h, w) at slot values p (N, slots)."""
        im, kind = self.im, self.kind
        q = [v.view(-1, 1, 1, 1) for v in p.unbind(1)]
        hu, hv, w = self.nodes
        if kind == SKY_FLAT:
            return (im.area * q[0] + 0 * (self.i + self.j))[:, 0]
        if kind == SKY_PLANE:
            du, dv = self.j - 0.5 * im.W, self.i - 0.5 * im.H
            dx, dy = im.A[0, 0] * du + im.A[0, 1] * dv, im.A[1, 0] * du + im.A[1, 1] * dv
            return (im.area * (q[0] + q[1] * dx + q[2] * dy))[:, 0]
        Ai = np.linalg.inv(im.A)
        wx, wy = q[0] - im.origin[0], q[1] - im.origin[1]
        du = self.j + hu - (Ai[0, 0] * wx + Ai[0, 1] * wy)
        dv = self.i + hv - (Ai[1, 0] * wx + Ai[1, 1] * wy)
        if kind == PSF_STAR:
            P = torch.tensor(im.psf, dtype=torch.float64, device="cuda")
            P = torch.nn.functional.pad(P / P.sum(), (1, 1, 1, 1))
            x, y = (torch.broadcast_tensors(du + im.h + 1, dv + im.h + 1))
            fx, fy = x.detach().floor().clamp(0, im.K), y.detach().floor().clamp(0, im.K)
            tx, ty = (x - fx), (y - fy)
            inside = (x > 0) & (x < im.K + 1) & (y > 0) & (y < im.K + 1)
            a, b = fy.long(), fx.long()
            top, bot = P[a, b] * (1 - tx) + P[a, b + 1] * tx, P[a + 1, b] * (1 - tx) + P[a + 1, b + 1] * tx
            return q[2][:, 0] * (w * torch.where(inside, top * (1 - ty) + bot * ty, torch.zeros_like(top))).sum(1)
        dx, dy = im.A[0, 0] * du + im.A[0, 1] * dv, im.A[1, 0] * du + im.A[1, 1] * dv
        c, s = torch.cos(q[3]), torch.sin(q[3])
        r2 = (dx * c + dy * s) ** 2 + ((dy * c - dx * s) / q[2]) ** 2
        if kind in (SERSIC, EXPONENTIAL):
            if kind == SERSIC:
                n, Re, Ie = q[4], q[5], q[6]
                b = self.b.view(-1, 1, 1, 1) + self.db.view(-1, 1, 1, 1) * (n - self.n0.view(-1, 1, 1, 1))
            else:
                n, Re, Ie, b = 1.0, q[4], q[5], _BN1
            f = Ie * torch.exp(-b * (((r2 + 1e-8 * im.area) / Re ** 2) ** (0.5 / n) - 1))
        elif kind == GAUSSIAN:
            f = q[5] / (2 * math.pi * q[4] ** 2 * q[2]) * torch.exp(-0.5 * r2 / q[4] ** 2)
        else:
            f = q[6] * (q[4] - 1) / (math.pi * q[5] ** 2 * q[2]) * (1 + r2 / q[5] ** 2) ** (-q[4])
        return im.area * (w * f).sum(1)


_BN1 = _bn_root(1.0)


def _batches(pr, image, theta, order, exact=True):
    found = {}
    for s in pr.sources:
        if s.image == image:
            found.setdefault((s.type, s.conv, s.box[1] - s.box[0], s.box[3] - s.box[2]), []).append(s)
    for (_, _, h, w), ss in found.items():
        most = max(1, (1 << 24) // (h * w * order * order))
        for k in range(0, len(ss), most):
            yield _Batch(pr, ss[k:k + most], theta, order, exact)


def _fast_len(n):
    while True:
        m = n
        for f in (2, 3, 5, 7):
            while m % f == 0:
                m //= f
        if m == 1:
            return n
        n += 1


def _convolve(x, psf):
    """Full linear convolution of the last two axes with a small kernel."""
    H, W = x.shape[-2] + psf.shape[0] - 1, x.shape[-1] + psf.shape[1] - 1
    n = (_fast_len(H), _fast_len(W))
    return torch.fft.irfft2(torch.fft.rfft2(x, s=n) * torch.fft.rfft2(psf, s=n), s=n)[..., :H, :W]


def _unit_psf(im):
    p = torch.tensor(im.psf, dtype=torch.float64, device="cuda")
    return p / p.sum()


def _model_images(pr, theta, order, exact=True):
    out = []
    for k, im in enumerate(pr.images):
        gal = torch.zeros(im.H + 2 * im.h, im.W + 2 * im.h, dtype=torch.float64, device="cuda")
        unc = torch.zeros(im.H, im.W, dtype=torch.float64, device="cuda")
        any_conv = False
        for b in _batches(pr, k, theta, order, exact):
            v = b.values(b.p)
            for s, x in zip(b.sources, v):
                o = im.h if s.conv else 0
                any_conv |= s.conv
                (gal if s.conv else unc)[s.box[0] + o:s.box[1] + o, s.box[2] + o:s.box[3] + o] += x
        if any_conv:
            unc += _convolve(gal, _unit_psf(im))[im.K - 1:im.H + im.K - 1, im.K - 1:im.W + im.K - 1]
        out.append(unc)
    return out


def _data(pr, c, seed):
    """Data, variance and mask of every image (float32, float32, uint8)."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))
    out = []
    for im, m in zip(pr.images, _model_images(pr, pr.theta, c["order"], exact=False)):
        var = (m.clamp(min=0) + im.floor) * im.var_scale
        z = torch.randn(im.H, im.W, generator=gen, device="cuda", dtype=torch.float64)
        mask = None
        if c["mask"] > 0:
            mask = (torch.rand(im.H, im.W, generator=gen, device="cuda") < c["mask"]).to(torch.uint8)
        out.append(((m + var.sqrt() * z).float(), var.float(), mask))
    return out


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def prepare(case, seed):
    c = case
    pr = _build(c, seed)
    images = []
    for im, (data, var, mask) in zip(pr.images, _data(pr, c, seed)):
        psf = None if im.psf is None else torch.tensor(im.psf, device="cuda")
        images.append(api.DeviceImage(im.H, im.W, im.A, im.origin, im.group, data, var, mask, psf, im.psf_pidx, im.psf_pfix))
    ctx = api.Context(c["precision"], quad_order=c["order"])
    ctx.set_problem(images, pr.sources, pr.theta.size)
    return SimpleNamespace(case=c, ctx=ctx, theta=torch.tensor(pr.start, device="cuda"),
                           lam=torch.full((pr.n_groups,), LAMBDA0, dtype=torch.float64, device="cuda"))


def run(state):
    c, ctx = state.case, state.ctx
    out = (lambda t: t) if c["precision"] == "f64" else (lambda t: t.float())
    if c["call"] == "eval":
        chi2, grad = ctx.eval(state.theta)
        return {"chi2": out(chi2), "grad": out(grad)}
    if c["call"] == "render":
        return {"model": ctx.render(state.theta)}
    if c["call"] == "adaptive":
        r = ctx.eval_adaptive(state.theta, model=True)
        return {"chi2": out(r["chi2"]), "model": r["model"]}
    if c["call"] == "shifted":
        chi2, model = ctx.eval_shifted(state.theta, model=True)
        return {"chi2": out(chi2), "model": model}
    if c["call"] == "normal":
        jtwr, (row_ptr, col_idx, vals) = ctx.normal_eq(state.theta)
        return {"jtwr": out(jtwr), "row_ptr": row_ptr, "col_idx": col_idx, "jtwj": out(vals)}
    theta, lam, chi2, _ = ctx.lm_iterate(state.theta, state.lam, c["iterations"])
    return {"theta": out(theta), "lambda": out(lam), "chi2": out(chi2)}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _area(b):
    return max(b[1] - b[0], 0) * max(b[3] - b[2], 0)


def _gram_flops(pr):
    """Products of the free columns of every two sources over the pixels both reach (one triangle)."""
    total = 0.0
    for k in range(len(pr.images)):
        ss = [s for s in pr.sources if s.image == k and s.free]
        if not ss:
            continue
        b, m = np.array([s.sup for s in ss]), np.array([len(s.free) for s in ss], dtype=float)
        for a in range(len(ss)):
            rows = np.minimum(b[a:, 1], b[a, 1]) - np.maximum(b[a:, 0], b[a, 0])
            cols = np.minimum(b[a:, 3], b[a, 3]) - np.maximum(b[a:, 2], b[a, 2])
            total += 2.0 * float((np.maximum(rows, 0) * np.maximum(cols, 0) * m[a:]).sum() * m[a])
    return total


def work(case):
    c = case
    pr = _build(c, 1)
    P, pixels = pr.theta.size, sum(im.H * im.W for im in pr.images)
    nodes = sum(_area(s.box) for s in pr.sources if s.type not in (SKY_FLAT, SKY_PLANE)) * c["order"] ** 2
    planes = sum(im.H * im.W for im in pr.images if im.K > 0)

    def transform(n):           # a convolution by real transforms there and back
        return 5.0 * n * math.log2(max(n, 2))

    columns = sum(transform(_area(s.sup)) * len(s.free) for s in pr.sources if s.conv)
    forward = 20.0 * nodes + transform(planes) + 6.0 * pixels
    backward = transform(planes) + 40.0 * nodes
    reads = pixels * (9 if c["mask"] > 0 else 8)
    size = 8 if c["precision"] == "f64" else 4
    if c["call"] in ("render", "adaptive", "shifted"):
        return {"bytes": pixels * size + (0 if c["call"] == "render" else reads) + 8 * P, "flops": forward}
    if c["call"] == "eval":
        return {"bytes": reads + 16 * P, "flops": forward + backward}
    if c["call"] == "normal":
        nnz = sum(len(s.free) ** 2 for s in pr.sources)
        return {"bytes": reads + 16 * P + 12 * nnz, "flops": forward + backward + columns + _gram_flops(pr)}
    n = c["iterations"]
    return {"bytes": reads + 24 * P, "flops": forward + n * (forward + backward + columns + _gram_flops(pr))}


# ---------------------------------------------------------------------------
# 64-bit results
# ---------------------------------------------------------------------------

class _Exact:
    def __init__(self, c, seed):
        self.c, self.pr = c, _build(c, seed)
        pr = self.pr
        self.P = pr.theta.size
        self.data = [(d.double(), torch.zeros_like(v.double()) if m is None else m.double(), v.double())
                     for d, v, m in _data(pr, c, seed)]
        self.group = np.full(self.P, -1)
        for s in pr.sources:
            for k in s.free:
                if self.group[s.pidx[k]] < 0:
                    self.group[s.pidx[k]] = pr.images[s.image].group

    def residuals(self, theta):
        """chi^2 per group and, per image, w r."""
        chi2, wr = np.zeros(self.pr.n_groups), []
        for im, m, (d, mask, var) in zip(self.pr.images, _model_images(self.pr, theta, self.c["order"]), self.data):
            w = (1 - mask) / var
            r = d - m
            chi2[im.group] += float((w * r * r).sum())
            wr.append(w * r)
        return chi2, wr

    def gradient(self, theta, wr):
        g = np.zeros(self.P)
        for k, im in enumerate(self.pr.images):
            adj = _convolve(wr[k], _unit_psf(im).flip(0, 1)) if im.K > 0 else None
            for b in _batches(self.pr, k, theta, self.c["order"]):
                p = b.p.clone().requires_grad_(True)
                o = im.h if b.sources[0].conv else 0
                a = adj if b.sources[0].conv else wr[k]
                cot = torch.stack([a[s.box[0] + o:s.box[1] + o, s.box[2] + o:s.box[3] + o] for s in b.sources])
                (d,) = torch.autograd.grad((b.values(p) * cot).sum(), p)
                for s, row in zip(b.sources, d.cpu().numpy()):
                    for slot in s.free:
                        g[s.pidx[slot]] += row[slot]
        return g

    def normal(self, theta):
        """J^T W J, dense on the device."""
        M = torch.zeros(self.P, self.P, dtype=torch.float64, device="cuda")
        side = 128
        for k, im in enumerate(self.pr.images):
            cols = []
            for b in _batches(self.pr, k, theta, self.c["order"]):
                free, conv = b.sources[0].free, b.sources[0].conv
                D = []
                for slot in free:
                    t = torch.zeros_like(b.p)
                    t[:, slot] = 1.0
                    D.append(torch.func.jvp(b.values, (b.p,), (t,))[1])
                D = torch.stack(D, 1)
                for s, x in zip(b.sources, D):
                    if conv:
                        full = _convolve(x, _unit_psf(im))
                        r, q = s.sup[0] - s.box[0] + im.h, s.sup[2] - s.box[2] + im.h
                        x = full[:, r:r + s.sup[1] - s.sup[0], q:q + s.sup[3] - s.sup[2]]
                    cols.append((s, x))
            _, mask, var = self.data[k]
            w = (1 - mask) / var
            for r0 in range(0, im.H, side):
                for c0 in range(0, im.W, side):
                    r1, c1 = min(r0 + side, im.H), min(c0 + side, im.W)
                    here = [(s, x) for s, x in cols if s.sup[0] < r1 and s.sup[1] > r0 and s.sup[2] < c1 and s.sup[3] > c0]
                    if not here:
                        continue
                    idx = [s.pidx[slot] for s, _ in here for slot in s.free]
                    J = torch.zeros(len(idx), r1 - r0, c1 - c0, dtype=torch.float64, device="cuda")
                    at = 0
                    for s, x in here:
                        a0, a1, b0, b1 = max(s.sup[0], r0), min(s.sup[1], r1), max(s.sup[2], c0), min(s.sup[3], c1)
                        part = x[:, a0 - s.sup[0]:a1 - s.sup[0], b0 - s.sup[2]:b1 - s.sup[2]]
                        J[at:at + len(x), a0 - r0:a1 - r0, b0 - c0:b1 - c0] = part
                        at += len(x)
                    G = (J * w[r0:r1, c0:c1]).flatten(1) @ J.flatten(1).T
                    i = torch.tensor(np.asarray(idx), device="cuda")
                    M.index_put_((i[:, None], i[None, :]), G, accumulate=True)
        return M

    def structure(self):
        """The stored entries: parameters of sources that reach a common 16 x 16 pixel tile of an image."""
        pattern = np.zeros((self.P, self.P), dtype=bool)
        for k in range(len(self.pr.images)):
            ss = [s for s in self.pr.sources if s.image == k and s.free and _area(s.sup) > 0]
            if not ss:
                continue
            t = np.array([(s.sup[0] // 16, (s.sup[1] - 1) // 16, s.sup[2] // 16, (s.sup[3] - 1) // 16) for s in ss])
            for a, s in enumerate(ss):
                meet = (t[:, 0] <= t[a, 1]) & (t[:, 1] >= t[a, 0]) & (t[:, 2] <= t[a, 3]) & (t[:, 3] >= t[a, 2])
                idx = np.array([ss[b].pidx[f] for b in np.nonzero(meet)[0] for f in ss[b].free])
                for f in s.free:
                    pattern[s.pidx[f], idx] = True
                    pattern[idx, s.pidx[f]] = True
        return np.nonzero(pattern)

    def bounds(self):
        lo, hi = np.full(self.P, -np.inf), np.full(self.P, np.inf)
        for s in self.pr.sources:
            box = {}
            if s.type <= MOFFAT:
                box[2] = (0.05, 1.0)
                box[4] = (0.36, 8.0) if s.type == SERSIC else (1.05, 50.0) if s.type == MOFFAT else (1e-3, np.inf)
                if s.type in (SERSIC, MOFFAT):
                    box[5] = (1e-3, np.inf)
            for k in s.free:
                if k in box:
                    lo[s.pidx[k]], hi[s.pidx[k]] = max(lo[s.pidx[k]], box[k][0]), min(hi[s.pidx[k]], box[k][1])
        return lo, hi

    def iterate(self, n):
        theta, lam = self.pr.start.copy(), np.full(self.pr.n_groups, LAMBDA0)
        lo, hi = self.bounds()
        chi2, wr = self.residuals(theta)
        for _ in range(n):
            M, g = self.normal(theta), self.gradient(theta, wr)
            D = M.diagonal().cpu().numpy().copy()
            for k in range(self.pr.n_groups):
                mine = self.group == k
                if mine.any():
                    D[mine] = np.maximum(D[mine], 1e-12 * D[mine].max())
            damped = M + torch.diag(torch.tensor(lam[self.group] * D, device="cuda"))
            step = torch.cholesky_solve(torch.tensor(g, device="cuda")[:, None], torch.linalg.cholesky(damped))[:, 0]
            trial = np.clip(theta + step.cpu().numpy(), lo, hi)
            c1, wr1 = self.residuals(trial)
            ok = np.isfinite(c1) & (c1 < chi2)
            theta = np.where(ok[self.group], trial, theta)
            lam = np.where(ok, np.maximum(lam / 9, 1e-12), np.minimum(lam * 11, 1e12))
            chi2 = np.where(ok, c1, chi2)
            wr = [b if ok[im.group] else a for im, a, b in zip(self.pr.images, wr, wr1)]
        return theta, lam, chi2


def exact(case, seed):
    c = case
    if c["call"] in ("adaptive", "shifted") or c["live_psf"]:
        return None
    pr = _build(c, seed)
    if c["call"] in ("normal", "lm"):   # about 20 seconds of float64 columns and products
        columns = sum(_area(s.sup) * len(s.free) * (c["order"] ** 2 + 20) for s in pr.sources)
        cost = max(c["iterations"], 1) * (columns / 4e8 + _gram_flops(pr) / 4e11)
        if pr.theta.size > 6000 or cost > 12:
            return None
    x = _Exact(c, seed)
    if c["call"] == "render":
        return {"model": _model_images(x.pr, x.pr.start, c["order"])}
    if c["call"] == "lm":
        theta, lam, chi2 = x.iterate(c["iterations"])
        return {"theta": theta, "lambda": lam, "chi2": chi2}
    chi2, wr = x.residuals(x.pr.start)
    g = x.gradient(x.pr.start, wr)
    if c["call"] == "eval":
        return {"chi2": chi2, "grad": -2.0 * g}
    rows, cols = x.structure()
    M = x.normal(x.pr.start)
    vals = M[torch.tensor(rows, device="cuda"), torch.tensor(cols, device="cuda")]
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=x.P))]).astype(np.int64)
    return {"jtwr": g, "row_ptr": row_ptr, "col_idx": cols.astype(np.int32), "jtwj": vals}
