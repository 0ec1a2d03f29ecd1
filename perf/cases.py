"""The work that users of this library have it do, as cases that can be timed and compared.

Every case goes through the public binding (paper_1002_1505_gb300.dda) with the state a user's
program holds: a context with its target, beams, Green tensor and polarizabilities, device vectors,
or a network.  Kinds:

  product  A P for all right-hand sides of a context: what a solve repeats
  solve    one whole dda_solve
  setup    what a new wavelength costs: beams, Green tensor, polarizability, incident field and the
           first product
  scatter  efficiencies, Mueller matrices and angular averages of solved polarizations
  net      the warm start's network: forward pass on the features of a target
  train    loss and gradient of one training batch of that network

Targets are ellipsoids (el), rectangular prisms (re) and hexagonal prisms (he) given as site lists.
"""
import math

import numpy as np
import torch

from paper_1002_1505_gb300 import dda as D

CIN, COUT, CH = 9, 6, (12, 24, 32, 48)
B1, B2, B3 = -1.8915316, 0.1648469, -1.7700004


def _case(kind, name=None, **kw):
    c = {"kind": kind}
    if name:
        c["name"] = name
    c.update(kw)
    return c


def _target(shape, nx, ny, nz, oris, mr, mi, x, pad=None, ncomp=1):
    c = {"shape": shape, "nx": nx, "ny": ny, "nz": nz, "oris": oris, "mr": mr, "mi": mi, "x": x, "ncomp": ncomp}
    c.update({"px": pad[0], "py": pad[1], "pz": pad[2]} if pad else {"px": 0, "py": 0, "pz": 0})
    return c


SPHERE = _target("el", 12, 12, 12, 1, 1.33, 0.01, 1.0)
ELLIPSOID = _target("el", 64, 48, 32, 1, 1.5, 0.1, 5.0, (128, 96, 64))
PRISM = _target("re", 48, 48, 48, 64, 1.7, 0.3, 8.0)
HEXAGON = _target("he", 111, 128, 160, 16, 1.33, 0.001, 20.0, (256, 256, 320))
RAGGED = _target("el", 45, 27, 37, 1, 2.1, 0.2, 4.0)
BLOCK = _target("re", 32, 64, 64, 1, 0.9656, 1.8628, 6.187304)


def listed():
    return [
        # the smallest call: the sphere of the accuracy tests, both polarizations; launches count
        _case("product", "product sphere12", dtype="c64", **SPHERE),
        # the guide-sized single-orientation run
        _case("product", "product ellipsoid64", dtype="c64", **ELLIPSOID),
        # an orientation average: 64 orientations x 2 polarizations in one batch
        _case("product", "product prism48 x128", dtype="c64", **PRISM),
        # the large target, 16 orientations x 2 polarizations (the benchmark's default)
        _case("product", "product hexprism160 x32", dtype="c64", **HEXAGON),
        # a target whose box is no convenient length and whose grid the library pads by itself, as
        # the random shapes of the warm start's training data
        _case("product", "product ragged", dtype="c64", **RAGGED),
        # the same in complex128: plain FP64 solves and their residuals
        _case("product", "product ragged c128", dtype="c128", **RAGGED),
        # the FP64-accurate product behind the true residual of every mixed solve
        _case("product", "residual ellipsoid64", dtype="df", **ELLIPSOID),
        # a whole solve, both polarizations, tight enough for six digits in the efficiencies
        _case("solve", "solve ellipsoid64", tol=1e-7, **ELLIPSOID),
        # one more wavelength of the same target
        _case("setup", "wavelength ellipsoid64", **ELLIPSOID),
        # the observables of the guide's worked example: 38 scattering directions and <cos>
        _case("scatter", "scattering block64", ndir=38, eta=0.5, **BLOCK),
        # the network's guess for the ellipsoid, both polarizations
        _case("net", "network 64x48x32 x2", nx=64, ny=48, nz=32, batch=2),
        # one training batch of the warm start's recipe: 16 samples on 16^3 grids
        _case("train", "training 16^3 x16", nx=16, ny=16, nz=16, batch=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product"] * 6 + ["solve", "setup", "scatter", "net", "train"])
    if kind in ("net", "train"):
        top = 48 if kind == "net" else 24
        dims = [8 * max(1, _log(rng, 8, top) // 8) for _ in range(3)]
        return _case(kind, nx=dims[0], ny=dims[1], nz=dims[2], batch=_log(rng, 1, 4 if kind == "net" else 16))
    lo, hi = (8, 100) if kind == "product" else (8, 48)
    dims = [_log(rng, lo, hi) for _ in range(3)]
    sites = dims[0] * dims[1] * dims[2]
    most = max(1, min(32, int(4e6 / sites))) if kind == "product" else 2
    t = _target(rng.choice(["el", "re", "he"]), *dims, oris=_log(rng, 1, most), mr=rng.uniform(1.1, 2.1),
                mi=rng.uniform(0.05, 0.5), x=rng.uniform(1.0, 6.0), ncomp=rng.choice([1, 1, 1, 2]))
    if kind == "product":
        dtype = rng.choice(["c64", "c64", "c64", "c128"])
        if dtype == "c128":
            t["oris"] = 1
        return _case(kind, dtype=dtype, **t)
    if kind == "solve":
        return _case(kind, tol=1e-7, **dict(t, oris=1, ncomp=1))
    if kind == "scatter":
        return _case(kind, ndir=_log(rng, 2, 90), eta=rng.uniform(0.5, 1.0), **t)
    return _case(kind, **t)


# ---------------------------------------------------------------- inputs
def _sites(c):
    """Sites (n, 3) as box indices, x fastest."""
    z, y, x = np.meshgrid(*(np.arange(c[a]) - (c[a] - 1) / 2.0 for a in ("nz", "ny", "nx")), indexing="ij")
    if c["shape"] == "re":
        keep = np.ones(x.shape, bool)
    elif c["shape"] == "el":
        keep = (2 * x / c["nx"]) ** 2 + (2 * y / c["ny"]) ** 2 + (2 * z / c["nz"]) ** 2 <= 1.0
    else:  # hexagonal cross section in x and y, vertices on y, stretched to the box
        keep = 2 * np.abs(y) / c["ny"] + np.abs(x) / c["nx"] <= 1.0
    ijk = np.argwhere(keep)[:, ::-1]
    return np.ascontiguousarray(ijk - ijk.min(axis=0), dtype=np.int32)


def _beams(c, seed):
    """Orientations (beta, Theta, Phi), uniform on the sphere."""
    rng = np.random.default_rng([seed, 1])
    n = c["oris"]
    return np.stack([rng.uniform(0, 2 * np.pi, n), np.arccos(rng.uniform(-1, 1, n)), rng.uniform(0, 2 * np.pi, n)], 1)


def _comps(c, n):
    return None if c["ncomp"] == 1 else (1 + np.arange(n) % c["ncomp"]).astype(np.int32)


def _indices(c, seed):
    """Refractive indices of the compositions: the case's, varied a little by the seed as over a wavelength."""
    f = 1.0 + 0.01 * np.random.default_rng([seed, 2]).uniform(-1, 1)
    m = complex(c["mr"] * f, c["mi"])
    return [m, m + 0.1][: c["ncomp"]]


def _kd(c, n, m, seed):
    aeff = (3.0 * n / (4.0 * np.pi)) ** (1.0 / 3.0)
    f = 1.0 + 0.01 * np.random.default_rng([seed, 3]).uniform(-1, 1)
    return f * min(c["x"] / aeff, 0.8 / max(abs(v) for v in m))


def _polarization(c, sites, seed):
    """Polarizations as a solve meets them: a wave through the target with noise on it, (2 oris, 3, n) complex128."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = len(sites)
    k = np.random.default_rng([seed, 4]).uniform(-0.3, 0.3, 3)
    ph = torch.as_tensor(sites, device="cuda", dtype=torch.float64) @ torch.as_tensor(k, device="cuda")
    wave = torch.polar(torch.ones_like(ph), ph).to(torch.complex64)
    p = torch.randn((2 * c["oris"], 3, n), dtype=torch.complex64, device="cuda", generator=g)
    return p.mul_(0.5).add_(wave)


def _context(c, seed):
    sites = _sites(c)
    m, ctx = _indices(c, seed), D.Context(0)
    ctx.dda_setup_target(sites, _comps(c, len(sites)))
    kd = _kd(c, len(sites), m, seed)
    ctx.dda_set_incident(kd, _beams(c, seed))
    ctx.dda_build_green_fft([c["px"], c["py"], c["pz"]] if c["px"] else None)
    ctx.dda_set_polarizability("GKDLDR", m)
    return ctx, sites, kd, m


def _dirs(c, seed):
    r = np.random.default_rng([seed, 5])
    return np.stack([np.linspace(0, np.pi, c["ndir"]), r.uniform(0, 2 * np.pi, c["ndir"])], 1)


def _net_shapes():
    c1, c2, c3, c4 = CH
    pairs = [(CIN, c1), (c1, c1), (c1, c2), (c2, c2), (c2, c3), (c3, c3), (c3, c4), (c4, c4), (c4 + c3, c3), (c3, c3),
             (c3 + c2, c2), (c2, c2), (c2 + c1, c1), (c1, c1)]
    return [(27, a, b) for a, b in pairs] + [(1, c1, COUT)]


def _net_params(seed):
    """He-initialised weights and small biases, layer by layer W [tap][in][out] then b."""
    r = np.random.default_rng([seed, 6])
    flat = []
    for t, a, b in _net_shapes():
        flat += [r.standard_normal(t * a * b) * math.sqrt(2.0 / (t * a)), 0.05 * r.standard_normal(b)]
    return np.concatenate(flat).astype(np.float32)


def _net_batch(c, seed):
    """Features of an ellipsoid filling the grid (occupancy, permittivity, incident wave), targets, mask."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    ax = [(torch.arange(c[a], device="cuda") - (c[a] - 1) / 2.0) for a in ("nz", "ny", "nx")]
    z, y, x = torch.meshgrid(*ax, indexing="ij")
    occ = (((2 * x / c["nx"]) ** 2 + (2 * y / c["ny"]) ** 2 + (2 * z / c["nz"]) ** 2) <= 1.0).float()
    B = c["batch"]
    k = torch.rand((B, 3), device="cuda", generator=g) * 0.6 - 0.3
    ph = k[:, 0, None, None, None] * x + k[:, 1, None, None, None] * y + k[:, 2, None, None, None] * z
    e = torch.rand((B, 3), device="cuda", generator=g) * 2 - 1
    eps = torch.rand((B, 2), device="cuda", generator=g)
    f = torch.zeros((B, c["nz"], c["ny"], c["nx"], CIN), device="cuda")
    f[..., 0] = occ
    f[..., 1:3] = occ[..., None] * eps[:, None, None, None, :]
    for a in range(3):
        f[..., 3 + 2 * a] = occ * e[:, a, None, None, None] * torch.cos(ph)
        f[..., 4 + 2 * a] = occ * e[:, a, None, None, None] * torch.sin(ph)
    t = 0.3 * torch.randn(f.shape[:4] + (COUT,), device="cuda", generator=g) + 0.5 * f[..., 3:9]
    return f.contiguous(), (t * occ[..., None]).contiguous(), occ.expand(B, -1, -1, -1).contiguous()


def prepare(case, seed):
    c = case
    if c["kind"] in ("net", "train"):
        net = D.UNet(0, None, CIN, COUT, CH, seed=0)
        net.dda_unet_set_params(_net_params(seed))
        f, t, mask = _net_batch(c, seed)
        return {"c": c, "net": net, "f": f, "t": t, "mask": mask, "y": torch.empty_like(t),
                "dims": (c["nx"], c["ny"], c["nz"])}
    ctx, sites, kd, m = _context(c, seed)
    s = {"c": c, "ctx": ctx}
    if c["kind"] == "product":
        p = _polarization(c, sites, seed)
        s["p"] = p if c["dtype"] == "c64" else p.to(torch.complex128)
        s["ap"] = torch.empty_like(s["p"])
    elif c["kind"] == "solve":
        s["p"] = torch.zeros((ctx.nrhs, 3, ctx.n), dtype=torch.complex128, device="cuda")
    elif c["kind"] == "scatter":
        s["p"] = _polarization(c, sites, seed).to(torch.complex128)
        s["dirs"] = _dirs(c, seed)
    else:
        s.update(kd=kd, m=m, beams=_beams(c, seed))
        s["e"] = torch.empty((ctx.nrhs, 3, ctx.n), dtype=torch.complex128, device="cuda")
        s["ap"] = torch.empty((ctx.nrhs, 3, ctx.n), dtype=torch.complex64, device="cuda")
    return s


def run(state):
    s, c = state, state["c"]
    if c["kind"] == "product":
        s["ctx"].dda_matvec(s["p"], s["ap"], double_float=c["dtype"] == "df")
        return s["ap"]
    if c["kind"] == "solve":
        s["ctx"].dda_solve(s["p"], solver="BICGSTAB", precision="MIXED", tol=c["tol"])
        return s["p"].to(torch.complex64)  # kept in single precision, as the tolerance is
    if c["kind"] == "setup":
        ctx = s["ctx"]
        ctx.dda_set_incident(s["kd"], s["beams"])
        ctx.dda_build_green_fft([c["px"], c["py"], c["pz"]] if c["px"] else None)
        ctx.dda_set_polarizability("GKDLDR", s["m"])
        ctx.dda_incident_field(s["e"])
        ctx.dda_matvec(s["e"].to(torch.complex64), s["ap"])
        return s["e"], s["ap"]
    if c["kind"] == "scatter":
        q, mueller = s["ctx"].dda_cross_sections(s["p"], s["dirs"])
        avg, _ = s["ctx"].dda_angular_averages(s["p"], c["eta"])
        return q, mueller, avg.astype(np.float32)  # the averages' phases are single precision
    if c["kind"] == "net":
        s["net"].dda_unet_forward(s["f"], s["y"], s["dims"])
        return s["y"]
    loss = s["net"].dda_unet_loss_grad(s["f"], s["t"], s["mask"], s["dims"])
    return loss, s["net"].dda_unet_get_params(1)


# ---------------------------------------------------------------- what a pass cannot do without
def _smooth(v):
    while True:
        q = v
        for f in (2, 3, 5):
            while q % f == 0:
                q //= f
        if q == 1 and v % 2 == 0:
            return v
        v += 1


def _pads(c, box):
    return (c["px"], c["py"], c["pz"]) if c["px"] else tuple(_smooth(2 * int(b)) for b in box)


def _product_work(c, n, box, size):
    """Bytes: P read, A P written, the interaction of the box's offsets once; flops: pruned transforms of
    three components there and back and the 3 x 3 multiply."""
    px, py, pz = _pads(c, box)
    nx, ny, nz = box
    fft = ny * nz * px * math.log2(px) + px * nz * py * math.log2(py) + px * py * pz * math.log2(pz)
    rhs = 2 * c["oris"]
    return 2 * rhs * 3 * n * size + 6 * nx * ny * nz * size, rhs * (6 * 5 * fft + 66 * px * py * pz)


def _net_flops(c):
    v = c["batch"] * c["nx"] * c["ny"] * c["nz"]
    level = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0]
    return sum(2 * t * a * b * v / 8 ** lv for (t, a, b), lv in zip(_net_shapes(), level))


def work(case):
    c = case
    if c["kind"] in ("net", "train"):
        v = c["batch"] * c["nx"] * c["ny"] * c["nz"]
        params = sum(t * a * b + b for t, a, b in _net_shapes())
        if c["kind"] == "net":
            return {"bytes": 4 * (v * (CIN + COUT) + params), "flops": _net_flops(c)}
        return {"bytes": 4 * (v * (CIN + COUT + 1) + 2 * params), "flops": 3 * _net_flops(c)}
    sites = _sites(c)
    n, box = len(sites), tuple(int(v) + 1 for v in sites.max(axis=0))
    rhs = 2 * c["oris"]
    if c["kind"] == "product":
        b, f = _product_work(c, n, box, 8 if c["dtype"] == "c64" else 16)
    elif c["kind"] == "solve":  # two products an iteration; about 20 iterations reach the tolerance
        b, f = _product_work(c, n, box, 8)
        b, f = 40 * b, 40 * f
    elif c["kind"] == "setup":
        b, f = _product_work(c, n, box, 8)
        px, py, pz = _pads(c, box)
        b, f = b + rhs * 3 * n * 16, f + 6 * 5 * px * py * pz * math.log2(px * py * pz) / 8
    else:
        dirs = len(_average_dirs(_kd(c, n, _indices(c, 0), 0) * (3.0 * n / (4.0 * np.pi)) ** (1.0 / 3.0), c["eta"]))
        b, f = rhs * 3 * n * 16, rhs * (dirs + c["ndir"]) * n * 24.0
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- the same in 64 bits, without the library
def _frame(ori):
    """x, y, z of the Lab Frame in the Target Frame (a1 = x_TF, a2 = y_TF)."""
    b, t, f = ori
    ct, st, cb, sb, cf, sf = np.cos(t), np.sin(t), np.cos(b), np.sin(b), np.cos(f), np.sin(f)
    return np.array([[ct, -st * cb, st * sb], [st * cf, ct * cb * cf - sb * sf, -(ct * sb * cf + cb * sf)],
                     [st * sf, ct * cb * sf + sb * cf, -(ct * sb * sf - cb * cf)]])


def _waves(oris, kd):
    """Per right-hand side: k and polarization in the Target Frame (e01 = y, e02 = x cross y = z)."""
    k, e = [], []
    for o in oris:
        f = _frame(o)
        k += [kd * f[0], kd * f[0]]
        e += [f[1], f[2]]
    return np.array(k), np.array(e)


def _inv_alpha(m, kd, k):
    eps, kh = m * m, k / kd
    cm = 4.0 * np.pi / 3.0 * (eps + 2) / (eps - 1) - 2j / 3 * kd ** 3
    return cm + (B1 + eps * B2 + eps * B3 * kh ** 2) * kd ** 2


class _Exact:
    """A of one case as FFT convolution in complex128."""

    def __init__(self, c, seed):
        self.sites = _sites(c)
        self.n = len(self.sites)
        self.m = _indices(c, seed)
        self.kd = kd = _kd(c, self.n, self.m, seed)
        self.oris = _beams(c, seed)
        self.k, self.e = _waves(self.oris, kd)
        box = self.sites.max(axis=0) + 1
        self.pad = P = _pads(c, box)
        off = [torch.tensor([o if o < b else (o - p if o > p - b else 0) for o in range(p)], dtype=torch.float64,
                            device="cuda") for p, b in zip(P, box)]
        ok = [torch.tensor([o < b or o > p - b for o in range(p)], device="cuda") for p, b in zip(P, box)]
        z, y, x = torch.meshgrid(off[2], off[1], off[0], indexing="ij")
        live = ok[2][:, None, None] & ok[1][None, :, None] & ok[0][None, None, :]
        r2 = x * x + y * y + z * z
        live &= r2 > 0
        r2 = torch.where(live, r2, torch.ones_like(r2))
        r = r2.sqrt()
        pref = torch.polar(live / r, kd * r)
        t2 = torch.complex(-1.0 / r2, kd * r / r2)
        h = (x / r, y / r, z / r)
        self.g = {}
        for a in range(3):
            for b in range(a, 3):
                hh, dl = h[a] * h[b], 1.0 if a == b else 0.0
                self.g[a, b] = self.g[b, a] = torch.fft.fftn(pref * (kd * kd * (hh - dl) + t2 * (3 * hh - dl)))
        s = torch.as_tensor(self.sites, device="cuda", dtype=torch.int64)
        self.at = (s[:, 2] * P[1] + s[:, 1]) * P[0] + s[:, 0]
        comp = _comps(c, self.n)
        self.comp = torch.as_tensor(np.zeros(self.n, np.int64) if comp is None else comp - 1, device="cuda")

    def alpha_inv(self, b):
        t = torch.as_tensor(np.array([_inv_alpha(m, self.kd, self.k[b]) for m in self.m]), device="cuda")
        return t[self.comp].T  # (3, n)

    def apply(self, b, p):
        shape = (self.pad[2], self.pad[1], self.pad[0])
        f = []
        for a in range(3):
            grid = torch.zeros(shape[0] * shape[1] * shape[2], dtype=torch.complex128, device="cuda")
            grid[self.at] = p[a]
            f.append(torch.fft.fftn(grid.view(shape)))
        out = self.alpha_inv(b) * p
        for a in range(3):
            out[a] += torch.fft.ifftn(sum(self.g[a, q] * f[q] for q in range(3))).reshape(-1)[self.at]
        return out

    def field(self, b):
        r = torch.as_tensor(self.sites, device="cuda", dtype=torch.float64)
        ph = r @ torch.as_tensor(self.k[b], device="cuda")
        return torch.as_tensor(self.e[b], device="cuda")[:, None] * torch.polar(torch.ones_like(ph), ph)

    def solve(self, b, tol=1e-11, most=2000):
        """Conjugate gradients for complex symmetric matrices (COCG)."""
        e = self.field(b)
        x, r = torch.zeros_like(e), e.clone()
        p, rho = r.clone(), (r * r).sum()
        for _ in range(most):
            v = self.apply(b, p)
            a = rho / (p * v).sum()
            x += a * p
            r -= a * v
            if float(r.norm() / e.norm()) <= tol:
                break
            new = (r * r).sum()
            p, rho = r + (new / rho) * p, new
        return x


def _average_dirs(x, eta):
    """(theta, phi, weight) of the guide's sampling of scattering directions."""
    t0 = 2 * np.pi / (1 + x)
    n = 1 + 2 * (3 + x) / eta * (1 + 1 / (np.pi + t0)) / (1 + t0 / (np.pi + t0) ** 2)
    n = max(3, int(round(n)))
    s = np.arange(n) * np.pi * (1 + 1 / (np.pi + t0)) / (n - 1)
    th = ((s - 1 - t0) + np.sqrt((1 + t0 - s) ** 2 + 4 * t0 * s)) / 2
    th[0], th[-1] = 0.0, np.pi
    out = []
    for j in range(n):
        nphi = 1 if j in (0, n - 1) else max(3, int(round(4 * np.pi * np.sin(th[j]) / (th[j + 1] - th[j - 1]))))
        if j == 0:
            w = 2 * np.pi * (1 - (1 + np.cos(th[1])) / 2)
        elif j == n - 1:
            w = 2 * np.pi * ((np.cos(th[j - 1]) - 1) / 2 + 1)
        else:
            w = np.pi / nphi * (np.cos(th[j - 1]) - np.cos(th[j + 1]))
        out += [(th[j], 2 * np.pi * i / nphi, w) for i in range(nphi)]
    return np.array(out)


def _lab(t, f):
    n = np.stack([np.cos(t), np.sin(t) * np.cos(f), np.sin(t) * np.sin(f)], -1)
    th = np.stack([-np.sin(t), np.cos(t) * np.cos(f), np.cos(t) * np.sin(f)], -1)
    ph = np.stack([0 * t, -np.sin(f), np.cos(f)], -1)
    return n, th, ph


def _far(x, p, n_tf):
    """F = sum_j P_j exp(-i k n.r_j), (directions, 3)."""
    r = torch.as_tensor(x.sites, device="cuda", dtype=torch.float64)
    out = []
    for n in torch.as_tensor(n_tf, device="cuda").split(64):
        ph = -x.kd * (n @ r.T)
        out.append(torch.polar(torch.ones_like(ph), ph) @ p.T)
    return torch.cat(out).cpu().numpy()


def _scatter_exact(c, seed):
    x, k = _Exact(c, seed), 0.0
    k, P = x.kd, _polarization(c, x.sites, seed).to(torch.complex128)
    aeff = (3.0 * x.n / (4.0 * np.pi)) ** (1.0 / 3.0)
    geo = np.pi * aeff ** 2
    dirs, av = _dirs(c, seed), _average_dirs(k * aeff, c["eta"])
    nd, td, fd = _lab(dirs[:, 0], dirs[:, 1])
    na = _lab(av[:, 0], av[:, 1])[0]
    q, avg, mue = [], [], []
    for o in range(c["oris"]):
        f, amp = _frame(x.oris[o]), []
        for b in (2 * o, 2 * o + 1):
            ep = complex((x.field(b).conj() * P[b]).sum())
            ab = float(((-x.alpha_inv(b).imag - 2.0 / 3.0 * k ** 3) * P[b].abs() ** 2).sum())
            ext, sca = 4 * np.pi * k * ep.imag / geo, 4 * np.pi * k * ab / geo
            q.append([ext, sca, ext - sca, 2 * np.pi * k * ep.real / geo])
            F = _far(x, P[b], na @ f)
            tr = F - (na @ f) * np.sum((na @ f) * F, -1, keepdims=True)
            dc = k ** 4 * np.sum(np.abs(tr) ** 2, -1) * av[:, 2]
            ct = np.cos(av[:, 0])
            avg.append([dc.sum() / geo, (dc * ct).sum() / dc.sum(), (dc * ct * ct).sum() / dc.sum(),
                        *(dc @ na / dc.sum())])
            F = _far(x, P[b], nd @ f)
            amp.append([k ** 3 * np.sum((td @ f) * F, -1), k ** 3 * np.sum((fd @ f) * F, -1)])
        # e01 = y, e02 = z: a = 1, b = 0, c = 0, d = 1
        (f11, f21), (f12, f22) = amp
        cp, sp = np.cos(dirs[:, 1]), np.sin(dirs[:, 1])
        s1, s2 = -1j * (-f21 * sp + f22 * cp), -1j * (f11 * cp + f12 * sp)
        s3, s4 = 1j * (-f11 * sp + f12 * cp), 1j * (f21 * cp + f22 * sp)
        h, a1, a2, a3, a4 = np.conj, *(np.abs(v) ** 2 for v in (s1, s2, s3, s4))
        mue.append(np.stack([
            (a1 + a2 + a3 + a4) / 2, (a2 - a1 + a4 - a3) / 2, (s2 * h(s3) + s1 * h(s4)).real,
            (s2 * h(s3) - s1 * h(s4)).imag, (a2 - a1 + a3 - a4) / 2, (a1 + a2 - a3 - a4) / 2,
            (s2 * h(s3) - s1 * h(s4)).real, (s2 * h(s3) + s1 * h(s4)).imag, (s2 * h(s4) + s1 * h(s3)).real,
            (s2 * h(s4) - s1 * h(s3)).real, (s1 * h(s2) + s3 * h(s4)).real, (s2 * h(s1) + s4 * h(s3)).imag,
            (s4 * h(s2) + s1 * h(s3)).imag, (s4 * h(s2) - s1 * h(s3)).imag, (s1 * h(s2) - s3 * h(s4)).imag,
            (s1 * h(s2) - s3 * h(s4)).real], -1).reshape(-1, 4, 4))
    return np.array(q), np.array(mue), np.array(avg)


def _net_exact(c, seed):
    """The network in float64 without any rounding of its operands; loss and gradient for a training case."""
    F = torch.nn.functional
    theta = torch.as_tensor(_net_params(seed), device="cuda").double().requires_grad_(c["kind"] == "train")
    f, t, mask = _net_batch(c, seed)
    layers, o = [], 0
    for taps, a, b in _net_shapes():
        w = theta[o:o + taps * a * b].view(*((3, 3, 3) if taps == 27 else (1, 1, 1)), a, b).permute(4, 3, 0, 1, 2)
        layers.append((w, theta[o + taps * a * b:o + taps * a * b + b]))
        o += taps * a * b + b
    it = iter(layers)

    def two(v):
        for _ in range(2):
            w, b = next(it)
            v = F.relu(F.conv3d(v, w, b, padding=1))
        return v

    up = torch.nn.Upsample(scale_factor=2, mode="nearest")
    s1 = two(f.double().permute(0, 4, 1, 2, 3))
    s2 = two(F.avg_pool3d(s1, 2))
    s3 = two(F.avg_pool3d(s2, 2))
    v = two(F.avg_pool3d(s3, 2))
    for skip in (s3, s2, s1):
        v = two(torch.cat([up(v), skip], 1))
    w, b = next(it)
    y = F.conv3d(v, w, b).permute(0, 2, 3, 4, 1)
    if c["kind"] == "net":
        return y
    loss = (((y - t) ** 2).sum(-1) * mask).sum() / (mask.double().sum() * COUT)
    return float(loss.detach()), torch.autograd.grad(loss, theta)[0]


def exact(case, seed):
    c = case
    if c["kind"] in ("net", "train"):
        return _net_exact(c, seed)
    if c["kind"] == "scatter":
        return _scatter_exact(c, seed)
    x = _Exact(c, seed)
    rhs = range(2 * c["oris"])
    if c["kind"] == "product":
        p = _polarization(c, x.sites, seed)
        out = torch.empty(p.shape, dtype=torch.complex128, device="cuda")
        for b in rhs:
            out[b] = x.apply(b, p[b].to(torch.complex128))
        return out
    if c["kind"] == "solve":
        return torch.stack([x.solve(b) for b in rhs])
    e = torch.stack([x.field(b) for b in rhs])
    return e, torch.stack([x.apply(b, e[b].to(torch.complex64).to(torch.complex128)) for b in rhs])
