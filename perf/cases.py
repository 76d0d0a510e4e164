"""Workloads of the SFFT library, each one pass through its public entry points.

A case is a plain dict: the entry point (``kind``), the image size, the fit
(kernel half-width, polynomial degrees or B-splines, photometric ratio), the
precision and how many pairs or systems go into one pass.  ``listed`` gives
the fixed cases, ``draw`` more of the same ranges, ``prepare`` the inputs and
the handles a program keeps (plan, server, captured batch), ``run`` one pass,
``work`` the bytes and operations no implementation can avoid, and ``exact``
the same outputs from torch FFTs and a dense solve in 64 bits.

The inputs are star fields: point sources with a power-law flux distribution,
two blended elliptical PSFs that differ between the reference and the science
image, a sloping sky, Poisson and read noise, and transients on the science
image alone.

What is returned: a mixed-precision pair returns its difference image, the
product of the pipeline (float32; coefficients, matrix and status stay in the
plan, where the C call keeps them when it is given none of these buffers).
The plain FP64 path returns coefficients and difference image or matrix and
right-hand side, all float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

FWHM = 1.0 / (2.0 * math.sqrt(2.0 * math.log(2.0)))


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


# ---------------------------------------------------------------------------
# cases

def _case(kind, n0, n1, w, dk, db, const=True, precision="mixed", spline="", masked=False, count=1, name=None):
    c = {"kind": kind, "n0": n0, "n1": n1, "w": w, "dk": dk, "db": db, "const": const, "precision": precision,
         "spline": spline, "masked": masked, "count": count}
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # a small cutout in the plain FP64 path, double images: launches and latency
        _case("pair", 256, 256, 4, 0, 0, precision="fp64", name="pair256_fp64"),
        # one ordinary single-CCD pair: linear kernel and sky, free photometric ratio
        _case("pair", 1024, 1024, 6, 1, 1, const=False, name="pair1024"),
        # the wide-field pair alone: latency of one pair of the benchmark's workload
        _case("pair", 4096, 4096, 8, 2, 2, name="pair4096"),
        # a whole CCD of 2046 x 4094 pixels, not powers of two, crowded field:
        # saturated pixels are found and masked for the fit
        _case("pair", 2046, 4094, 6, 2, 1, masked=True, name="ccd2046x4094"),
        # kernel and sky varying as B-splines instead of polynomials
        _case("pair", 2048, 2048, 8, 0, 0, spline="1,1,2,1", name="bspline2048"),
        # a survey's stream of wide-field pairs through the server, eight in flight
        _case("serve", 4096, 4096, 8, 2, 2, count=8, name="serve4096"),
        # uneven sectors (512..2048 px, a fit each) captured once and replayed
        _case("sectors", 512, 2048, 8, 2, 2, count=16, name="sectors16"),
        # the normal equations alone in FP64, rows that are not a power of two
        _case("build", 1000, 1024, 5, 1, 1, precision="fp64", name="build_fp64"),
        # one built system of the wide-field fit (1735 unknowns)
        _case("solve", 1024, 1024, 8, 2, 2, name="solve1735"),
        # eight built systems of different fits solved together
        _case("solve", 768, 768, 8, 2, 2, count=8, name="solve_batch8"),
        # a known kernel applied to another pair of the field, odd row count
        _case("subtract", 3001, 2048, 7, 2, 1, name="subtract3001"),
        # noise decorrelation of a difference image of four and four co-added exposures
        _case("decorrelate", 4096, 4096, 8, 2, 2, count=4, name="decorrelate_coadd"),
    ]


def _size(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    r = rng.random()
    if r < 0.3:  # powers of two are common sizes
        return 1 << int(round(math.log2(n)))
    return n | 1 if r < 0.6 else n


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "pair", "serve", "sectors", "build", "solve", "solve", "subtract",
                       "decorrelate"])
    w, dk, db, const = rng.randint(4, 8), rng.randint(0, 2), rng.randint(0, 2), rng.random() < 0.6
    precision, spline, masked, count = "mixed", "", False, 1
    n0 = _size(rng, 256, 4096)
    n1 = n0 if rng.random() < 0.4 else max(256, min(4096, int(n0 * rng.uniform(0.5, 2.0))))
    if kind == "pair":
        r = rng.random()
        if r < 0.25:
            precision = "fp64"
            n0, n1 = min(n0, 1024), min(n1, 1024)
        elif r < 0.45:
            spline = rng.choice(["1,1,2,1", "2,0,1,1", "1,0,1,0", "2,1,2,0"])
            dk = db = 0
            n0, n1 = min(n0, 2048), min(n1, 2048)
        elif r < 0.7:
            masked = True
    elif kind == "serve":
        count = rng.randint(2, 8)
    elif kind == "sectors":
        n0, n1 = 512, rng.randint(1024, 2048)
        count = rng.randint(8, 16)
    elif kind == "build":
        precision = "fp64"
        n0, n1 = min(n0, 1024), min(n1, 1024)
    elif kind == "solve":
        n0 = n1 = rng.randint(600, 1024)
        count = rng.choice([1, 2, 4, 8])
    elif kind == "decorrelate":
        count = rng.choice([0, 2, 4])
    return _case(kind, n0, n1, w, dk, db, const, precision, spline, masked, count)


def _spline(c):
    return tuple(int(v) for v in c["spline"].split(",")) if c["spline"] else None


def _parts(c):
    """The pairs or systems of one pass: (n0, n1, w, dk, db, const) of each.
    A batch of sectors has square sizes spread over [n0, n1] and a fit each; a
    batch of systems has different fits; the pairs of a server share one."""
    base = (c["n0"], c["n1"], c["w"], c["dk"], c["db"], c["const"])
    if c["kind"] == "sectors":
        r = np.random.RandomState(c["n1"] + c["count"])
        return [(n, n, int(r.randint(4, 9)), int(r.randint(0, 3)), int(r.randint(0, 3)), c["const"])
                for n in (int(v) for v in r.randint(c["n0"], c["n1"] + 1, c["count"]))]
    if c["kind"] == "solve" and c["count"] > 1:
        return [(c["n0"], c["n1"], max(4, c["w"] - k // 2), max(1, c["dk"]) if k % 2 == 0 else 1, c["db"], c["const"])
                for k in range(c["count"])]
    return [base] * (c["count"] if c["kind"] == "serve" else 1)


# ---------------------------------------------------------------------------
# inputs

def _coords(n, dev):
    x = torch.arange(n, dtype=torch.float64, device=dev)
    return (2.0 * x - (n - 1)) / max(n - 1, 1)


def _psf_hat(n0, n1, fwhm, ellip, dev):
    """Transform (real FFT layout) of a unit elliptical Gaussian, long axis at 30 degrees."""
    f0 = 2 * math.pi * torch.fft.fftfreq(n0, dtype=torch.float64, device=dev)[:, None]
    f1 = 2 * math.pi * torch.fft.rfftfreq(n1, dtype=torch.float64, device=dev)[None, :]
    s2 = (fwhm * FWHM) ** 2
    a, b = s2 / (1.0 - ellip), s2 * (1.0 - ellip)
    ca, sa = math.cos(math.pi / 6), math.sin(math.pi / 6)
    u, v = ca * f0 + sa * f1, ca * f1 - sa * f0
    return torch.exp(-0.5 * (a * u * u + b * v * v))


def _images(n0, n1, seed, dtype):
    """One reference and science image: a star per 800 pixels, PSFs that widen
    from the centre to the edge, transients on the science image alone."""
    dev = _dev()
    r = np.random.RandomState(seed % (1 << 31))
    gen = torch.Generator(device=dev).manual_seed(seed)
    ns, nt = max(8, n0 * n1 // 800), max(1, 50 * n0 * n1 // (4096 * 4096))

    def points(num, flux, edge=None):
        img = np.zeros((n0, n1))
        x, y = r.uniform(0, n0, num), r.uniform(0, n1, num)
        near, far = img, np.zeros((n0, n1))
        rad = ((2 * x / n0 - 1) ** 2 + (2 * y / n1 - 1) ** 2) / 2
        ix, iy = x.astype(int), y.astype(int)
        fx, fy = x - ix, y - iy
        for dx, wx in ((0, 1 - fx), (1, fx)):  # sub-pixel positions by bilinear weights
            for dy, wy in ((0, 1 - fy), (1, fy)):
                at = ((ix + dx) % n0, (iy + dy) % n1)
                np.add.at(near, at, flux * wx * wy * (1 - rad))
                np.add.at(far, at, flux * wx * wy * rad)
        return [torch.fft.rfft2(torch.from_numpy(v).to(dev)) for v in (near, far)]

    u = r.uniform(0, 1, ns)
    flux = (1e2 ** -1.5 - u * (1e2 ** -1.5 - 2e4 ** -1.5)) ** (-1 / 1.5)  # brighter ones saturate
    stars, trans = points(ns, flux), points(nt, r.uniform(1e3, 1e4, nt))
    xt, yt = _coords(n0, dev)[:, None], _coords(n1, dev)[None, :]

    def image(layers, near, far, ellip, sky):
        hat = layers[0] * _psf_hat(n0, n1, near, 0.0, dev) + layers[1] * _psf_hat(n0, n1, far, ellip, dev)
        img = torch.fft.irfft2(hat, s=(n0, n1)) + sky
        img = torch.poisson(img.clamp(min=0.0), generator=gen)
        noise = torch.randn((n0, n1), dtype=torch.float64, device=dev, generator=gen)
        return (img + 5.0 * noise).to(dtype).contiguous()

    ref = image(stars, 2.5, 3.0, 0.1, 100.0)
    both = [a + b for a, b in zip(stars, trans)]
    sci = image(both, 3.5, 4.5, 0.2, 100.0 + 20 * xt * xt + 10 * yt * yt + 5 * xt * yt)
    return ref, sci


SATURATION, GROW = 1500.0, 5


def _saturation(ref, sci):
    bad = ((ref >= SATURATION) | (sci >= SATURATION)).to(torch.float32)[None, None]
    grown = torch.nn.functional.max_pool2d(bad, 2 * GROW + 1, stride=1, padding=GROW)[0, 0]
    return (grown == 0).to(torch.uint8)


def _coadd(count, seed):
    """Homogenisation kernels of `count` exposures: 7 x 7 Gaussians, and their noise."""
    r = np.random.RandomState((seed + 7) % (1 << 31))
    k = torch.arange(-3, 4, dtype=torch.float64)
    out = []
    for _ in range(count):
        g = torch.exp(-(k[:, None] ** 2 + k[None, :] ** 2) / (2 * r.uniform(0.8, 1.6) ** 2))
        out.append(g / g.sum() / count)
    return torch.stack(out).to(_dev()).contiguous(), [float(v) for v in r.uniform(4.0, 8.0, count)]


# ---------------------------------------------------------------------------
# the fit in 64 bits: torch FFTs, the Gram matrix of the shifted basis images,
# a dense solve

def _bspline_functions(n, deg, interior, dev):
    """Clamped uniform B-splines of one axis by the Cox-de Boor recursion, [K][n]."""
    x = _coords(n, "cpu").numpy()
    t = np.concatenate([[-1.0] * deg, np.linspace(-1.0, 1.0, interior + 2), [1.0] * deg])
    last = len(t) - deg - 2
    fun = [((x >= t[i]) & (x < t[i + 1])).astype(float) for i in range(len(t) - 1)]
    fun[last] = ((x >= t[last]) & (x <= t[last + 1])).astype(float)
    for d in range(1, deg + 1):
        new = []
        for i in range(len(t) - 1 - d):
            v = np.zeros(n)
            if t[i + d] > t[i]:
                v += (x - t[i]) / (t[i + d] - t[i]) * fun[i]
            if t[i + d + 1] > t[i + 1]:
                v += (t[i + d + 1] - x) / (t[i + d + 1] - t[i + 1]) * fun[i + 1]
            new.append(v)
        fun = new
    return [torch.from_numpy(f).to(dev) for f in fun]


def _powers(d):
    return [(t - j, j) for t in range(d + 1) for j in range(t + 1)]


class _Fit64:
    """Terms, unknowns and transforms of one fit, in 64 bits."""

    def __init__(self, n0, n1, w, dk, db, const, spline):
        dev = _dev()
        self.n0, self.n1, self.w = n0, n1, w
        self.L1 = 2 * w + 1
        self.L, self.c = self.L1 ** 2, (self.L1 ** 2 - 1) // 2
        if spline:
            fx, fy = (_bspline_functions(n, spline[0], spline[1], dev) for n in (n0, n1))
            bx, by = (_bspline_functions(n, spline[2], spline[3], dev) for n in (n0, n1))
            self.terms = [(a, b) for a in fx for b in fy]
            self.back = [(a, b) for a in bx for b in by]
            self.keep = [[o for o in range(self.L) if not const or o != self.c] for _ in self.terms]
            if const:
                one = [torch.ones(n, dtype=torch.float64, device=dev) for n in (n0, n1)]
                self.terms.insert(0, tuple(one))
                self.keep.insert(0, [self.c])
        else:
            xt, yt = _coords(n0, dev), _coords(n1, dev)
            self.terms = [(xt ** i, yt ** j) for i, j in _powers(dk)]
            self.back = [(xt ** p, yt ** q) for p, q in _powers(db)]
            self.keep = [[o for o in range(self.L) if t == 0 or not const or o != self.c]
                         for t in range(len(self.terms))]
        self.n = sum(len(k) for k in self.keep) + len(self.back)

    def _hats(self, img):
        return [torch.fft.rfft2(f[:, None] * g[None, :] * img) for f, g in self.terms]

    def _lags(self, a, b, h):
        """Sum_x a(x) b(x + rho) for |rho| <= h, [2h+1][2h+1], of two real transforms."""
        full = torch.fft.irfft2(a.conj() * b, s=(self.n0, self.n1))
        k = torch.arange(-h, h + 1, device=full.device)
        return full[(k % self.n0)[:, None], (k % self.n1)[None, :]]

    def system(self, ref, sci, mask=None):
        ref, sci = ref.double(), sci.double()
        if mask is not None:
            ref, sci = ref * mask, sci * mask
        dev, w, L1, L, c = ref.device, self.w, self.L1, self.L, self.c
        hats, sh = self._hats(ref), torch.fft.rfft2(sci)
        B = torch.eye(L, dtype=torch.float64, device=dev)  # delta basis: shifted minus unshifted
        B[:, c] -= 1.0
        B[c, c] = 1.0
        o = torch.arange(L, device=dev)
        d0 = (o // L1)[:, None] - (o // L1)[None, :] + 2 * w
        d1 = (o % L1)[:, None] - (o % L1)[None, :] + 2 * w
        at = [torch.tensor(k, device=dev) for k in self.keep]
        start = np.cumsum([0] + [len(k) for k in self.keep])
        nkern = int(start[-1])
        M = torch.zeros((self.n, self.n), dtype=torch.float64, device=dev)
        rhs = torch.zeros(self.n, dtype=torch.float64, device=dev)
        for t in range(len(hats)):
            rows = slice(int(start[t]), int(start[t + 1]))
            for u in range(t, len(hats)):
                block = B @ self._lags(hats[t], hats[u], 2 * w)[d0, d1] @ B.T
                block = block[at[t]][:, at[u]]
                cols = slice(int(start[u]), int(start[u + 1]))
                M[rows, cols] = block
                M[cols, rows] = block.T
            rhs[rows] = (B @ self._lags(hats[t], sh, w).reshape(-1))[at[t]]
        for s, (f, g) in enumerate(self.back):
            img = f[:, None] * g[None, :]
            bh = torch.fft.rfft2(img)
            for t in range(len(hats)):
                rows = slice(int(start[t]), int(start[t + 1]))
                v = (B @ self._lags(hats[t], bh, w).reshape(-1))[at[t]]
                M[rows, nkern + s] = v
                M[nkern + s, rows] = v
            for s2, (f2, g2) in enumerate(self.back):
                M[nkern + s, nkern + s2] = (f * f2).sum() * (g * g2).sum()
            rhs[nkern + s] = (img * sci).sum()
        return M, rhs

    def solve(self, M, rhs):
        d = M.diagonal().rsqrt()
        A = d[:, None] * M * d[None, :]
        f = torch.linalg.cholesky(A)
        x = d * torch.cholesky_solve((d * rhs)[:, None], f)[:, 0]
        return x + d * torch.cholesky_solve((d * (rhs - M @ x))[:, None], f)[:, 0]

    def kernels(self, x):
        """Per term the kernel image [L1][L1] in the plain basis."""
        out, at = [], 0
        for k in self.keep:
            v = torch.zeros(self.L, dtype=torch.float64, device=x.device)
            v[torch.tensor(k, device=x.device)] = x[at:at + len(k)]
            v[self.c] = 2 * v[self.c] - v.sum()
            out.append(v.reshape(self.L1, self.L1))
            at += len(k)
        return out

    def kernel_hat(self, k):
        """Real transform of a centred kernel image on the image's grid."""
        h0, h1 = k.shape[0] // 2, k.shape[1] // 2
        img = torch.zeros((self.n0, self.n1), dtype=torch.float64, device=k.device)
        a = torch.arange(-h0, h0 + 1, device=k.device) % self.n0
        b = torch.arange(-h1, h1 + 1, device=k.device) % self.n1
        img[a[:, None], b[None, :]] = k
        return torch.fft.rfft2(img)

    def difference(self, ref, sci, x):
        ref, sci = ref.double(), sci.double()
        model = sum(h * self.kernel_hat(k) for h, k in zip(self._hats(ref), self.kernels(x)))
        out = sci - torch.fft.irfft2(model, s=(self.n0, self.n1))
        for (f, g), b in zip(self.back, x[self.n - len(self.back):]):
            out -= b * f[:, None] * g[None, :]
        return out

    def decorrelate(self, x, diff, ss, sr, G=None, H=None):
        """Noise decorrelation with the kernel at the centre of the field; G, H
        with noise ss, sr: the co-added form."""
        wt = [float(_mid(f) * _mid(g)) for f, g in self.terms]
        k2 = self.kernel_hat(sum(a * k for a, k in zip(wt, self.kernels(x)))).abs() ** 2
        if G is None:
            den = ss ** 2 + sr ** 2 * k2
        else:
            den = sum(s ** 2 * self.kernel_hat(g).abs() ** 2 for s, g in zip(ss, G))
            den = den + k2 * sum(s ** 2 * self.kernel_hat(g).abs() ** 2 for s, g in zip(sr, H))
        q = torch.sqrt(den[0, 0] / den)
        return torch.fft.irfft2(torch.fft.rfft2(diff.double()) * q, s=(self.n0, self.n1))


def _mid(f):
    """A polynomial term's value at the field centre, coordinate 0: 1 for the
    constant (all ones), 0 for the others."""
    return 1.0 if bool((f == 1.0).all()) else 0.0


# ---------------------------------------------------------------------------
# states, passes

def _fit(c, part):
    return _Fit64(*part, _spline(c))


def _seeds(c, seed):
    return [seed * 131 + 17 * k + 1 for k in range(len(_parts(c)))]


def _pair_inputs(c, part, seed):
    ref, sci = _images(part[0], part[1], seed, torch.float64 if c["precision"] == "fp64" else torch.float32)
    return ref, sci


def _plan(c, part):
    from paper_2109_09334_gb300 import SfftPlan
    n0, n1, w, dk, db, const = part
    return SfftPlan(n0, n1, w, w, dk, db, const, dtype="float64" if c["precision"] == "fp64" else "float32",
                    precision=c["precision"], spline=_spline(c))


def prepare(case, seed):
    c, kind = case, case["kind"]
    parts, seeds = _parts(c), _seeds(c, seed)
    s = {"case": c}
    if kind == "solve":  # systems as a build leaves them, made here from other images
        s["plans"] = [_plan(c, p) for p in parts]
        made = [_fit(c, p).system(*_pair_inputs(c, p, k)) for p, k in zip(parts, seeds)]
        s["M"], s["rhs"] = [m for m, _ in made], [r for _, r in made]
        s["x"] = [torch.empty_like(r) for r in s["rhs"]]
        return s
    imgs = [_pair_inputs(c, p, k) for p, k in zip(parts, seeds)]
    s["ref"], s["sci"] = [a for a, _ in imgs], [b for _, b in imgs]
    if kind == "serve":
        from paper_2109_09334_gb300 import SfftServer
        n0, n1, w, dk, db, const = parts[0]
        s["server"] = SfftServer(n0, n1, w, w, dk, db, const, depth=c["count"], batch=c["count"])
        s["D"] = [torch.empty_like(r) for r in s["ref"]]
        s["last"] = None
        return s
    if kind == "sectors":
        from paper_2109_09334_gb300 import SfftBatch
        s["plans"] = [_plan(c, p) for p in parts]
        for p in s["plans"]:
            p.solve_panel = 64
        s["batch"] = SfftBatch(s["plans"], s["ref"], s["sci"], solve_group=8)
        return s
    s["plan"] = _plan(c, parts[0])
    if kind == "pair":
        s["D"] = torch.empty_like(s["ref"][0])
        s["mask"] = torch.empty(s["D"].shape, dtype=torch.uint8, device=s["D"].device) if c["masked"] else None
    elif kind in ("subtract", "decorrelate"):
        fit = _fit(c, parts[0])
        s["x"] = fit.solve(*fit.system(s["ref"][0], s["sci"][0]))
        if kind == "decorrelate":
            s["diff"] = fit.difference(s["ref"][0], s["sci"][0], s["x"]).to(torch.float32)
            if c["count"]:
                s["G"], s["sG"] = _coadd(c["count"], seed)
                s["H"], s["sH"] = _coadd(c["count"], seed + 1)
            del s["ref"], s["sci"]
            s["out"] = torch.empty_like(s["diff"])
        else:  # the kernel found on one pair, applied to the next
            s["ref"][0], s["sci"][0] = _pair_inputs(c, parts[0], seeds[0] + 5)
    return s


def run(state):
    from paper_2109_09334_gb300 import binding
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "pair":
        plan, ref, sci = s["plan"], s["ref"][0], s["sci"][0]
        if c["precision"] == "fp64":
            D, x, _, _, _ = plan.run_pair(ref, sci, out=s["D"])
            return {"D": D, "x": x}
        if s["mask"] is None:
            binding.sfft_run_pair(plan.handle, ref, sci, None, None, None, None, None, s["D"], plan.stream)
            return {"D": s["D"]}
        binding.sfft_saturation_mask(ref, sci, SATURATION, SATURATION, GROW, s["mask"], stream=plan.stream)
        binding.sfft_run_pair(plan.handle, ref, sci, s["mask"], None, None, None, None, s["D"], plan.stream)
        return {"D": s["D"], "mask": s["mask"]}
    if kind == "serve":
        srv = s["server"]
        if s["last"] is not None:
            srv.poll(s["last"])  # releases the requests of the pass before
        for ref, sci, D in zip(s["ref"], s["sci"], s["D"]):
            s["last"] = srv.submit(ref, sci, diff=D)[0]
        srv.stream_wait(s["last"])
        return {"D": s["D"]}
    if kind == "sectors":
        s["batch"].launch()
        return {"D": s["batch"].D}
    if kind == "build":
        M, rhs = s["plan"].build_system(s["ref"][0], s["sci"][0])
        return {"M": M, "rhs": rhs}
    if kind == "solve":
        if c["count"] == 1:
            return {"x": [s["plans"][0].solve(s["M"][0], s["rhs"][0])[0]]}
        binding.sfft_solve_batch([p.handle for p in s["plans"]], s["M"], s["rhs"], s["x"], None, s["plans"][0].stream)
        return {"x": s["x"]}
    if kind == "subtract":
        return {"D": s["plan"].subtract(s["ref"][0], s["sci"][0], s["x"])}
    if c["count"]:
        return {"out": s["plan"].decorrelate_coadd(s["x"], s["diff"], s["G"], s["sG"], s["H"], s["sH"], out=s["out"])}
    return {"out": s["plan"].decorrelate(s["x"], s["diff"], 5.0, 6.0, out=s["out"])}


def exact(case, seed):
    c, kind = case, case["kind"]
    parts, seeds = _parts(c), _seeds(c, seed)
    if kind == "solve":
        out = []
        for p, k in zip(parts, seeds):
            fit = _fit(c, p)
            out.append(fit.solve(*fit.system(*_pair_inputs(c, p, k))))
        return {"x": out}
    if kind in ("serve", "sectors"):
        out = []
        for p, k in zip(parts, seeds):
            fit, (ref, sci) = _fit(c, p), _pair_inputs(c, p, k)
            out.append(fit.difference(ref, sci, fit.solve(*fit.system(ref, sci))))
        return {"D": out}
    fit, (ref, sci) = _fit(c, parts[0]), _pair_inputs(c, parts[0], seeds[0])
    if kind == "build":
        M, rhs = fit.system(ref, sci)
        return {"M": M, "rhs": rhs}
    mask = _saturation(ref, sci) if c["masked"] else None
    x = fit.solve(*fit.system(ref, sci, mask))
    if kind == "subtract":
        return {"D": fit.difference(*_pair_inputs(c, parts[0], seeds[0] + 5), x)}
    D = fit.difference(ref, sci, x)
    if kind == "decorrelate":
        D = D.to(torch.float32)
        if not c["count"]:
            return {"out": fit.decorrelate(x, D, 6.0, 5.0)}
        (G, sG), (H, sH) = _coadd(c["count"], seed), _coadd(c["count"], seed + 1)
        return {"out": fit.decorrelate(x, D, sG, sH, G, H)}
    if c["precision"] == "fp64":
        return {"D": D, "x": x}
    return {"D": D} if mask is None else {"D": D, "mask": mask}


def work(case):
    """Images, systems and results each moved once; transforms of the images
    that enter the fit (2.5 N log2 N each, forward and back), the products of
    their spectra, and a Cholesky factorisation."""
    c, kind = case, case["kind"]
    size = 8 if c["precision"] == "fp64" else 4
    nbytes = flops = 0.0
    sp = _spline(c)
    for n0, n1, w, dk, db, const in _parts(c):
        L, P = (2 * w + 1) ** 2, float(n0 * n1)
        if sp:
            K, nb = (sp[0] + sp[1] + 1) ** 2, (sp[2] + sp[3] + 1) ** 2
            nk, n = K + int(const), K * (L - int(const)) + int(const) + nb
        else:
            nk, nb = (dk + 1) * (dk + 2) // 2, (db + 1) * (db + 2) // 2
            n = (nk * (L - 1) + 1 if const else nk * L) + nb
        fft = 2.5 * P * math.log2(P)
        products = (nk * (nk + 1) / 2 + nk) * 4 * P
        if kind in ("pair", "serve", "sectors"):
            nbytes += 3 * size * P + (P if c["masked"] else 0)
            flops += (nk + 2) * fft + products + n ** 3 / 3 + 4 * nk * P
        elif kind == "build":
            nbytes += 2 * size * P + 8.0 * n * n + 8 * n
            flops += (nk + 1) * fft + products
        elif kind == "solve":
            nbytes += 8.0 * n * n + 16 * n
            flops += n ** 3 / 3
        elif kind == "subtract":
            nbytes += 3 * size * P + 8 * n
            flops += (nk + 2) * fft + 4 * nk * P
        else:
            nbytes += 2 * size * P + 8 * n
            flops += 2 * fft + 2 * P
    return {"bytes": nbytes, "flops": flops}
