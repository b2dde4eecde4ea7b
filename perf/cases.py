"""Workloads of the SPECT projector library, one dict each: what a user's program calls.

`listed()` covers the range of the repository's own configurations (64x64x32 with an
11x11 PSF, 128x128x80 with 37x37, the batching sizes 64..160, the large serving case
192x192x128), both directions (A, A'), the EM updates built on them, the gradient of an
EM update, ordered subsets and batches, and the plan options (full PSF, view-dependent
PSF, three-pass rotation, low-memory and recomputing plans).  `draw` gives more cases
of the same ranges.

Keys of a case
  op       forward | back | em | train | osem | batch
  nx nz nview px pz
  psf      "sep" (separable factors) or "full" (a stack that is not separable)
  orbit    True: every view has its own PSF
  plan     "default" | "lowmem" | "recompute" | "3pass"
  tune     True: the program lets the library time its launch shapes once
  niter    EM iterations of one call
  subsets  ordered subsets (osem)
  sizes    "nx x nz x nview x psf, ..." (batch)
"""
import math

import numpy as np
import torch

from paper_2301_09710_gb300 import SpectBatch, SpectPlan
from paper_2301_09710_gb300.autograd import em_update
from paper_2301_09710_gb300.osem import OSEM

FWHM_TO_SIGMA = 1.0 / (2.0 * math.sqrt(2.0 * math.log(2.0)))
BETA = 0.3  # weight of the regulariser in the training case


def _case(name, op, nx, nz, nview, px, pz, **more):
    c = {"name": name, "op": op, "nx": nx, "nz": nz, "nview": nview, "px": px, "pz": pz, "psf": "sep",
         "orbit": False, "plan": "default", "tune": False, "niter": 1}
    c.update(more)
    return c


def listed():
    return [
        # the smallest operator that the tests pin against the dense matrix: one A, all latency and launches
        _case("forward-16", "forward", 16, 8, 8, 5, 5),
        # the small configuration, reconstructed: two MLEM iterations a call, as the serving loop enqueues them
        _case("em-64", "em", 64, 32, 64, 11, 11, niter=2),
        # the benchmark workload, tuned once as the benchmark does: one MLEM iteration
        _case("em-128", "em", 128, 80, 128, 37, 37, tune=True),
        # measurements simulated at the largest size of the batching workload
        _case("forward-160", "forward", 160, 96, 120, 29, 29),
        # back-projection of a non-circular orbit: every view has its own PSF
        _case("back-orbit", "back", 128, 80, 120, 37, 37, orbit=True),
        # a ragged volume (no size divides anything) with px != pz
        _case("em-odd", "em", 99, 53, 60, 21, 15),
        # the large serving request
        _case("em-192", "em", 192, 128, 128, 37, 37),
        # a measured PSF that does not factorise
        _case("em-full-psf", "em", 96, 64, 60, 21, 21, psf="full"),
        # the other rotation of the paper
        _case("em-3pass", "em", 128, 64, 60, 21, 21, plan="3pass"),
        # a plan held small (many plans on a device)
        _case("em-lowmem", "em", 96, 64, 60, 21, 21, plan="lowmem"),
        # one regularised EM update of an unrolled network, forward and backward
        _case("train-96", "train", 96, 64, 64, 21, 21),
        # reconstructions of different sizes as one batch
        _case("batch-6", "batch", 0, 0, 0, 0, 0, niter=2,
              sizes="64x32x60x11,96x48x90x21,128x64x60x29,64x80x120x11,96x96x60x37,128x32x90x21"),
    ]


def draw(rng):
    """One more case of the same ranges, no costlier than the largest listed one."""
    while True:
        op = rng.choice(["forward", "back", "em", "em", "em", "train", "osem", "batch"])
        lim = 0.6 * _cost(_case("", "em", 192, 128, 128, 37, 37))
        if op == "batch":
            sizes = []
            for _ in range(rng.randint(2, 6)):
                sizes.append("%dx%dx%dx%d" % (_log(rng, 24, 160), _log(rng, 8, 96), _log(rng, 16, 128),
                                              2 * rng.randint(1, 18) + 1))
            c = _case("", "batch", 0, 0, 0, 0, 0, sizes=",".join(sizes), niter=rng.choice([1, 2, 4]))
        else:
            px = 2 * rng.randint(1, 18) + 1
            pz = px if rng.random() < 0.6 else 2 * rng.randint(1, 18) + 1
            c = _case("", op, _log(rng, 16, 192), _log(rng, 5, 128), _log(rng, 8, 128), px, pz)
            kind = rng.choice(["sep", "sep", "sep", "full", "lowmem", "recompute", "3pass"])
            if kind == "full":
                c["psf"] = "full"
            elif kind != "sep":
                c["plan"] = kind
            if kind == "lowmem" and rng.random() < 0.4:
                c["px"] = c["pz"] = 2 * rng.randint(19, 25) + 1  # wider than the fused kernels take
            c["orbit"] = kind == "sep" and rng.random() < 0.25
            if op == "em":
                c["niter"] = rng.choice([1, 1, 2])
                c["tune"] = kind == "sep" and c["nx"] <= 128 and rng.random() < 0.2
            if op == "osem":
                c["subsets"] = rng.choice([2, 4])
        del c["name"]
        if _cost(c) <= lim:
            return c


def _log(rng, lo, hi):
    """A size spread evenly over its logarithm, odd ones among them."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _members(case):
    """The single reconstructions of a batch, as cases of their own."""
    out = []
    for s in case["sizes"].split(","):
        nx, nz, nview, p = (int(t) for t in s.split("x"))
        out.append(_case("", "em", nx, nz, nview, p, p, niter=case["niter"]))
    return out


def _cost(case):
    """About how long a pass takes, in FP32 operations of the fused kernels."""
    if case["op"] == "batch":
        return sum(_cost(c) for c in _members(case))
    f = work(case)["flops"]
    return f * (12.0 if case["plan"] == "lowmem" else 1.0)


def work(case):
    """Bytes: each input read once, each output written once.  Operations, per voxel and view of
    one A or A': the blur 2(px+pz) (2 px pz for a full PSF), the rotation 8 (16 for three
    passes' eight taps), the attenuation and the sum 2."""
    if case["op"] == "batch":
        w = [work(c) for c in _members(case)]
        return {"bytes": sum(t["bytes"] for t in w), "flops": sum(t["flops"] for t in w)}
    nx, nz, nview, px, pz = (case[k] for k in ("nx", "nz", "nview", "px", "pz"))
    vol, proj = nx * nx * nz, nx * nz * nview
    taps = (px + pz if case["psf"] == "sep" else px * pz) * nx * (nview if case["orbit"] else 1)
    per = 2.0 * (px + pz if case["psf"] == "sep" else px * pz) + (16 if case["plan"] == "3pass" else 8) + 2
    one = per * vol * nview
    base = vol + taps  # mu and the PSF
    op, n = case["op"], case["niter"]
    if op in ("forward", "back"):
        return {"bytes": 4.0 * (base + vol + proj), "flops": one}
    if op == "train":  # x, y, rbar, s, u, g in; the update and two gradients out; A, A' and both transposed
        return {"bytes": 4.0 * (base + 7 * vol + 2 * proj), "flops": 4 * one}
    return {"bytes": 4.0 * (base + 3 * vol + 2 * proj), "flops": 2 * n * one}  # x, s, y, rbar in, x out


# ------------------------------------------------------------------ inputs
def _ellipsoid(grid, centre, semi, phi=0.0):
    i, j, k = (g - c for g, c in zip(grid, centre))
    c, s = math.cos(phi), math.sin(phi)
    return ((c * i + s * j) / semi[0]) ** 2 + ((c * j - s * i) / semi[1]) ** 2 + (k / semi[2]) ** 2 <= 1.0


def _phantom(nx, nz, rng, dev):
    """Activity, attenuation (per mm) and body: a body with organs, hot lesions, lungs and a spine."""
    r = lambda n: torch.arange(n, device=dev, dtype=torch.float32)  # noqa: E731
    grid = (r(nx)[None, None, :], r(nx)[None, :, None], r(nz)[:, None, None])
    c, ck = 0.5 * (nx - 1), 0.5 * (nz - 1)
    body = _ellipsoid(grid, (c, c, ck), (0.42 * nx, 0.30 * nx, 0.55 * nz)).expand(nz, nx, nx)
    x = body.float()
    for n in range(16):
        semi = rng.uniform(0.04, 0.14, 3) * (nx, nx, nz)
        a, d = rng.uniform(0, 2 * math.pi), 0.3 * nx * math.sqrt(rng.uniform())
        m = _ellipsoid(grid, (c + d * math.cos(a), c + d * math.sin(a), rng.uniform(0.2, 0.8) * (nz - 1)),
                       np.maximum(semi, 0.7), rng.uniform(0, math.pi))
        value = rng.uniform(0.3, 3.0) if n < 13 else rng.uniform(4.0, 8.0)
        x = torch.where(m & body, torch.full_like(x, value), x)
    mu = 0.015 * body.float()
    for side in (-1, 1):
        m = _ellipsoid(grid, (c + side * 0.2 * nx, c, 0.7 * (nz - 1)), (0.12 * nx, 0.14 * nx, 0.25 * nz + 0.5))
        mu = torch.where(m & body, torch.full_like(mu, 0.005), mu)
    m = _ellipsoid(grid, (c, c + 0.2 * nx, ck), (0.05 * nx + 0.5, 0.05 * nx + 0.5, 0.6 * nz))
    mu = torch.where(m & body, torch.full_like(mu, 0.030), mu)
    return x.contiguous(), mu.contiguous(), body.contiguous()


def _gauss(size, sigma, dev):
    """Rows of unit-sum Gaussians of the given widths."""
    t = torch.arange(size, device=dev, dtype=torch.float64) - (size - 1) // 2
    g = torch.exp(-0.5 * (t / sigma[..., None]) ** 2)
    return g / g.sum(-1, keepdim=True)


def _psf(case, rng, dev):
    """PSF factors (nvp, ny, px), (nvp, ny, pz), or a stack (nvp, ny, pz, px) that does not
    factorise: Gaussians that widen with the distance from the detector (plane ny-1)."""
    nx, px, pz = case["nx"], case["px"], case["pz"]
    nvp = case["nview"] if case["orbit"] else 1
    far = max(1.5, min(px, pz) / 4.0) * rng.uniform(0.9, 1.1)
    near = min(1.0, far) * rng.uniform(1.0, 1.5)
    gap = torch.zeros(nvp, 1, device=dev, dtype=torch.float64)
    if nvp > 1:
        gap[:, 0] = 0.04 * nx * torch.sin(2 * math.pi * torch.arange(nvp, device=dev) / nvp).abs()
    dist = (nx - 1 - torch.arange(nx, device=dev, dtype=torch.float64) + gap) / (nx - 1 + float(gap.max()))
    fwx = near + (far - near) * dist
    fwz = (0.8 * fwx + 0.3).clamp(near, max(near, far))
    sx, sz = fwx * FWHM_TO_SIGMA, fwz * FWHM_TO_SIGMA
    if case["psf"] == "sep":
        return _gauss(px, sx, dev).float(), _gauss(pz, sz, dev).float(), None
    a = (torch.arange(px, device=dev, dtype=torch.float64) - (px - 1) // 2)[None, None, None, :] / sx[..., None, None]
    b = (torch.arange(pz, device=dev, dtype=torch.float64) - (pz - 1) // 2)[None, None, :, None] / sz[..., None, None]
    p = torch.exp(-0.5 * (a * a + b * b - 0.6 * a * b)) + 0.02 / (1.0 + 0.3 * (a * a + b * b))  # tilted, with a tail
    return None, None, (p / p.sum((-2, -1), keepdim=True)).float()


def _counts(case, x, mu, dy, rng, dev):
    """Measured counts and a smooth background, about 6 counts a bin: the phantom turned, attenuated
    and summed by torch, blurred by one width, Poisson noise on top."""
    nz, nx, nview = case["nz"], case["nx"], case["nview"]
    out = torch.empty(nview, nz, nx, device=dev)
    both = torch.stack([x, mu])  # (2, nz, ny, nx)
    lin = torch.linspace(-1, 1, nx, device=dev) if nx > 1 else torch.zeros(1, device=dev)
    jj, ii = torch.meshgrid(lin, lin, indexing="ij")
    for l in range(nview):
        th = 2 * math.pi * l / nview
        g = torch.stack([math.cos(th) * ii + math.sin(th) * jj, math.cos(th) * jj - math.sin(th) * ii], -1)
        t = torch.nn.functional.grid_sample(both, g.expand(2, nx, nx, 2), mode="bilinear", padding_mode="zeros",
                                            align_corners=True)
        att = t[1].flip(1).cumsum(1).flip(1) - 0.5 * t[1]
        out[l] = (t[0] * torch.exp(-dy * att)).sum(1)
    k = _gauss(9, torch.tensor(1.5, dtype=torch.float64), "cpu").tolist()
    pad = torch.nn.functional.pad(out, (4, 4))
    out = sum(k[a] * pad[..., a:a + nx] for a in range(9))
    scale = 6.0 / float(out.mean())
    out *= scale
    rbar = torch.full_like(out, 0.6) * torch.linspace(0.8, 1.2, nx, device=dev)
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(rng.integers(1 << 30)))
    return torch.poisson(out + rbar, generator=gen), rbar, scale, gen


def _inputs(case, seed):
    dev = torch.device("cuda")
    rng = np.random.default_rng([seed, case["nx"], case["nz"], case["nview"]])
    dy = 4.8 * 128 / case["nx"]
    x, mu, body = _phantom(case["nx"], case["nz"], rng, dev)
    fx, fz, psf = _psf(case, rng, dev)
    y, rbar, scale, gen = _counts(case, x, mu, dy, rng, dev)
    x *= scale
    x0 = body.float() * float(x.mean())
    d = {"x": x, "mu": mu, "dy": dy, "fx": fx, "fz": fz, "psf": psf, "y": y, "rbar": rbar, "x0": x0}
    if case["op"] == "train":
        d["u"] = x0 * (0.5 + torch.rand(x0.shape, generator=gen, device=dev))
        d["g"] = torch.randn(x0.shape, generator=gen, device=dev)
    return d


def _plan(case, d):
    p = SpectPlan(case["nx"], case["nz"], case["nview"], mu=d["mu"], dy=d["dy"], psf=d["psf"], fx=d["fx"], fz=d["fz"],
                  low_memory=case["plan"] == "lowmem", recompute_attenuation=case["plan"] == "recompute",
                  rotation="3pass" if case["plan"] == "3pass" else "bilinear")
    if case["tune"]:
        p.autotune()
    return p


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        members = _members(case)
        ds = [_inputs(c, seed * 31 + n) for n, c in enumerate(members)]
        plans = [_plan(c, d) for c, d in zip(members, ds)]
        for p in plans:
            p.sensitivity()
        return {"case": case, "plans": plans, "batch": SpectBatch(plans), "x0": [d["x0"] for d in ds],
                "x": [d["x0"].clone() for d in ds], "y": [d["y"] for d in ds], "rbar": [d["rbar"] for d in ds]}
    d = _inputs(case, seed)
    d["case"] = case
    if op == "osem":
        m = case["subsets"]
        d["osem"] = OSEM(case["nx"], case["nz"], case["nview"], m, mu=d["mu"], dy=d["dy"], psf=d["psf"], fx=d["fx"],
                         fz=d["fz"], low_memory=case["plan"] == "lowmem",
                         recompute_attenuation=case["plan"] == "recompute",
                         rotation="3pass" if case["plan"] == "3pass" else "bilinear")
        d["ys"], d["rs"] = d["osem"].split(d["y"]), d["osem"].split(d["rbar"])
        for p in d["osem"].plans:
            p.sensitivity()
        return d
    d["p"] = _plan(case, d)
    if op in ("em", "train"):
        d["s"] = d["p"].sensitivity()
    return d


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "forward":
        return s["p"].forward(s["x"])
    if op == "back":
        return s["p"].back(s["y"])
    if op == "em":
        return s["p"].em_step(s["x0"].clone(), s["y"], s["rbar"], niter=case["niter"])
    if op == "osem":
        return s["osem"].step(s["x0"].clone(), s["ys"], s["rs"], niter=case["niter"])
    if op == "batch":
        for x, x0 in zip(s["x"], s["x0"]):
            x.copy_(x0)
        return s["batch"].em_step(s["x"], s["y"], s["rbar"], niter=case["niter"])
    x, u = s["x0"].detach().requires_grad_(), s["u"].detach().requires_grad_()
    x1 = em_update(x, s["y"], s["rbar"], s["p"], s["s"], u, BETA)
    gx, gu = torch.autograd.grad(x1, (x, u), s["g"])
    return x1.detach(), gx, gu


def tolerance(case):
    """FP32 results of positive sums.  Against 64 bits the library is seen at 3e-8 to 1.3e-7 (2-norm; one or
    two EM updates, A, A', the gradients); another order of its sums moves it as much.  Every further EM update
    adds as much again."""
    n = case["niter"] * (case.get("subsets", 1) if case["op"] == "osem" else 1)
    return {"rel": 5e-7 * n, "max": 2e-5 * n}


# ------------------------------------------------------------------ 64-bit values
class _Exact:
    """A and A' of one geometry in 64 bits, from their definitions: per view a sparse rotation (its taps
    as index and weight arrays), the attenuation, the blur with replicate padding, the depth sum."""

    def __init__(self, case, d, views=None):
        self.case, self.nx, self.nz = case, case["nx"], case["nz"]
        self.dev = d["mu"].device
        self.mu = d["mu"].double().reshape(self.nz, -1)
        self.dy = float(np.float32(d["dy"]))
        f = lambda t: None if t is None else t.double()  # noqa: E731
        self.fx, self.fz, self.psf = f(d["fx"]), f(d["fz"]), f(d["psf"])
        self.views = list(range(case["nview"])) if views is None else [int(v) for v in views]

    def _taps(self, l):
        """Stages of the rotation: each a list of (source pixel, weight) over the nx*nx pixels."""
        n, th = self.nx, 2 * math.pi * l / self.case["nview"]
        c = 0.5 * (n - 1)
        r = torch.arange(n, device=self.dev, dtype=torch.float64)
        j, i = torch.meshgrid(r, r, indexing="ij")
        q = round(th / (math.pi / 2))
        near = abs(th / (math.pi / 2) - q) < 1e-12

        def line(axis, pos):  # linear interpolation along one axis, zeros outside
            lo = torch.floor(pos)
            out = []
            for o, w in ((lo, 1 - (pos - lo)), (lo + 1, pos - lo)):
                ok = (o >= 0) & (o < n)
                o = o.clamp(0, n - 1)
                idx = (j * n + o) if axis == 0 else (o * n + i)
                out.append((idx.long().reshape(-1), (w * ok).reshape(-1)))
            return out

        if self.case["plan"] == "3pass":
            phi = th - q * (math.pi / 2)
            t, s = math.tan(phi / 2), math.sin(phi)
            si, sj = [(i, j), (j, n - 1 - i), (n - 1 - i, n - 1 - j), (n - 1 - j, i)][q % 4]
            one = [((sj * n + si).long().reshape(-1), torch.ones(n * n, device=self.dev, dtype=torch.float64))]
            return [one, line(0, i + t * (j - c)), line(1, j - s * (i - c)), line(0, i + t * (j - c))]
        ct, st = math.cos(th), math.sin(th)
        if near:
            ct, st = [(1.0, 0.0), (0.0, 1.0), (-1.0, 0.0), (0.0, -1.0)][q % 4]
        xs, ys = c + ct * (i - c) + st * (j - c), c - st * (i - c) + ct * (j - c)
        x0, y0 = torch.floor(xs), torch.floor(ys)
        taps = []
        for dj in (0, 1):
            for di in (0, 1):
                a, b = x0 + di, y0 + dj
                w = (xs - x0 if di else 1 - (xs - x0)) * (ys - y0 if dj else 1 - (ys - y0))
                ok = (a >= 0) & (a < n) & (b >= 0) & (b < n)
                taps.append(((b.clamp(0, n - 1) * n + a.clamp(0, n - 1)).long().reshape(-1), (w * ok).reshape(-1)))
        return [taps]

    @staticmethod
    def _turn(stages, x):
        for taps in stages:
            x = sum(x[:, idx] * w for idx, w in taps)
        return x

    @staticmethod
    def _turn_t(stages, x):
        for taps in reversed(stages):
            out = torch.zeros_like(x)
            for idx, w in taps:
                out.index_add_(1, idx, x * w)
            x = out
        return x

    def _view(self, l):
        stages = self._taps(l)
        m = self._turn(stages, self.mu).reshape(self.nz, self.nx, self.nx)
        s = m.flip(1).cumsum(1).flip(1) - 0.5 * m
        return stages, torch.exp(-self.dy * s)

    def _band(self, f, n):
        """(ny, n, n) matrices of the 1D convolution with replicate padding."""
        p = f.shape[-1]
        out = torch.zeros(f.shape[0], n, n, device=self.dev, dtype=torch.float64)
        r = torch.arange(n, device=self.dev)
        for a in range(p):
            src = (r - a + (p - 1) // 2).clamp(0, n - 1)
            out[:, r, src] += f[:, a, None]  # one source per row: no index twice
        return out

    def _blur(self, l):
        v = l if self.case["orbit"] else 0
        if self.psf is None:
            if getattr(self, "_at", None) != v:
                self._at, self._bx, self._bz = v, self._band(self.fx[v], self.nx), self._band(self.fz[v], self.nz)
            return self._bx, self._bz
        if getattr(self, "_at", None) != v:
            pz, px = self.psf.shape[-2:]
            self._size = (self.nz + 2 * (pz - 1), self.nx + 2 * (px - 1))
            self._at, self._hat = v, torch.fft.rfft2(self.psf[v], s=self._size)
        return self._hat, None

    def _pads(self):
        pz, px = self.psf.shape[-2:]
        cz, cx = (pz - 1) // 2, (px - 1) // 2
        k = (torch.arange(self.nz + 2 * cz, device=self.dev) - cz).clamp(0, self.nz - 1)
        i = (torch.arange(self.nx + 2 * cx, device=self.dev) - cx).clamp(0, self.nx - 1)
        return k, i, cz, cx

    def forward(self, x):
        x = x.double().reshape(self.nz, -1)
        out = torch.empty(len(self.views), self.nz, self.nx, device=self.dev, dtype=torch.float64)
        for n, l in enumerate(self.views):
            stages, mb = self._view(l)
            w = (self._turn(stages, x).reshape(self.nz, self.nx, self.nx) * mb).permute(1, 0, 2)  # (ny, nz, nx)
            a, b = self._blur(l)
            if b is not None:
                t = torch.bmm(w, a.transpose(1, 2))
                out[n] = b.permute(1, 0, 2).reshape(self.nz, -1) @ t.reshape(-1, self.nx)
            else:
                k, i, cz, cx = self._pads()
                hat = torch.fft.rfft2(w[:, k][:, :, i], s=self._size)
                full = torch.fft.irfft2((hat * a).sum(0), s=self._size)
                out[n] = full[2 * cz:2 * cz + self.nz, 2 * cx:2 * cx + self.nx]
        return out

    def back(self, v):
        v = v.double()
        out = torch.zeros(self.nz, self.nx * self.nx, device=self.dev, dtype=torch.float64)
        for n, l in enumerate(self.views):
            stages, mb = self._view(l)
            a, b = self._blur(l)
            if b is not None:
                t = torch.matmul(torch.matmul(b.transpose(1, 2), v[n]), a)  # (ny, nz, nx)
            else:
                k, i, cz, cx = self._pads()
                z = torch.zeros(self._size, device=self.dev, dtype=torch.float64)
                z[2 * cz:2 * cz + self.nz, 2 * cx:2 * cx + self.nx] = v[n]
                pad = torch.fft.irfft2(torch.fft.rfft2(z) * a.conj(), s=self._size)[:, :len(k), :len(i)]
                t = torch.zeros(self.nx, self.nz, len(i), device=self.dev, dtype=torch.float64).index_add_(1, k, pad)
                t = torch.zeros(self.nx, self.nz, self.nx, device=self.dev, dtype=torch.float64).index_add_(2, i, t)
            out += self._turn_t(stages, (t.permute(1, 0, 2) * mb).reshape(self.nz, -1))
        return out.reshape(self.nz, self.nx, self.nx)

    def em(self, x, y, rbar, s):
        yb = self.forward(x) + rbar.double()
        e = self.back(torch.where(yb > 0, y.double() / yb, torch.zeros_like(yb)))
        return torch.where(s > 0, x * e / s, torch.zeros_like(x))

    def ones(self):
        return torch.ones(len(self.views), self.nz, self.nx, device=self.dev, dtype=torch.float64)


def _exact_cost(case):
    """Operations of exact() in 64 bits."""
    if case["op"] == "batch":
        return sum(_exact_cost(c) for c in _members(case))
    nx, nz, nview = case["nx"], case["nz"], case["nview"]
    if case["psf"] == "sep":
        per = 2.0 * (nx + nz)
    else:
        per = 60.0 * (1 + 2 * case["px"] / nx) * (1 + 2 * case["pz"] / nz)
    n = {"forward": 1, "back": 1, "train": 5}.get(case["op"], 1 + 2 * case["niter"])
    return per * nx * nx * nz * nview * n


def exact(case, seed):
    if _exact_cost(case) > 4e12:
        return None
    if case["op"] == "batch":
        return [_exact_em(c, _inputs(c, seed * 31 + n)) for n, c in enumerate(_members(case))]
    d = _inputs(case, seed)
    op = case["op"]
    if op == "forward":
        return _Exact(case, d).forward(d["x"])
    if op == "back":
        return _Exact(case, d).back(d["y"])
    if op == "em":
        return _exact_em(case, d)
    if op == "osem":
        m = case["subsets"]
        parts = []
        for k in range(m):
            E = _Exact(case, d, range(k, case["nview"], m))
            parts.append((E, d["y"][k::m], d["rbar"][k::m], E.back(E.ones())))
        x = d["x0"].double()
        for _ in range(case["niter"]):
            for E, y, r, s in parts:
                x = E.em(x, y, r, s)
        return x
    # the regularised update and its gradient (implicit derivative of beta x1^2 + q x1 - x e = 0)
    E = _Exact(case, d)
    x, u, g = d["x0"].double(), d["u"].double(), d["g"].double()
    s = E.back(E.ones())
    yb = E.forward(x) + d["rbar"].double()
    ratio = d["y"].double() / yb
    e = E.back(ratio)
    dd = s - BETA * u
    q = torch.sqrt(dd * dd + 4 * BETA * x * e)
    x1 = torch.where(dd >= 0, 2 * x * e / (dd + q), (q - dd) / (2 * BETA))
    ge = E.forward(g * x / q)
    gx = g * e / q + E.back(-ge * ratio / yb)
    return x1, gx, g * BETA * x1 / q


def _exact_em(case, d):
    E = _Exact(case, d)
    s = E.back(E.ones())
    x = d["x0"].double()
    for _ in range(case["niter"]):
        x = E.em(x, d["y"], d["rbar"], s)
    return x
