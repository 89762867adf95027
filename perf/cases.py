"""Performance cases: the calls a user of the library makes, over the sizes they are made at.

Six kinds of work, each through the binding of the C entry points (``rb``):

* ``update``  one frequency-set update of a reconstruction (``rb_hf_update``): the call a sweep
              repeats, with the map, the measured data and the workspace resident;
* ``adjoint`` Born gradient and Hessian diagonal from given tables (``rb_born_adjoint``);
* ``forward`` Born data of a model perturbation from given tables (``rb_born_forward``);
* ``rays``    ray fans and the ray-model data at the receivers (``rb_trace_rays``,
              ``rb_ray_forward``);
* ``grid``    first-arrival tables and Green's functions (``rb_green_grid``);
* ``tof``     the time-of-flight initial guess (``rb_tof_invert``).

All inputs are made here, with torch, from the seed alone: breast-like phantoms (fat,
fibroglandular and lesion ellipses in water, smoothed), measured data with the straight-ray
traveltime, spreading and absorption of the true medium plus 1 % noise, and, for the single
operators, smooth first-arrival tables with holes outside the support.
"""
import math

import numpy as np
import torch

from paper_2511_16633_gb300 import rb

RADIUS = 0.110          # the ring's radius [m]
C_WATER = 1480.0
F_REF = 1.0e6
POWER_Y = 1.1
K_A = 11.512925464970229   # dB/cm -> Np/m
DEV = "cuda"


def listed():
    mixed, fp32 = "bf16x3", "fp32"
    return [
        # the smallest reconstruction of the tests: launches and latency
        dict(name="update_64el_64px", kind="update", n_elem=64, nx=64, ny=64, n_rays=64, n_freq=1, prec=mixed, f_lo=0.3, f_hi=0.3),
        # a 256-element ring on a coarse grid, three frequencies a set
        dict(name="update_256el_256px", kind="update", n_elem=256, nx=256, ny=256, n_rays=256, n_freq=3, prec=mixed, f_lo=0.3, f_hi=0.43),
        # the benchmark: 256 elements, 512 x 512 pixels, four frequencies a set
        dict(name="update_256el_512px", kind="update", n_elem=256, nx=512, ny=512, n_rays=256, n_freq=4, prec=mixed, f_lo=0.3, f_hi=0.45),
        # the in-vivo array: 512 elements with fans of 512 rays (two element passes)
        dict(name="update_512el_256px", kind="update", n_elem=512, nx=256, ny=256, n_rays=512, n_freq=4, prec=mixed, f_lo=0.5, f_hi=0.65),
        # plain FP32, which takes any ring up to 512 elements: an odd ring, a ragged grid
        dict(name="update_fp32_150el", kind="update", n_elem=150, nx=260, ny=243, n_rays=200, n_freq=2, prec=fp32, f_lo=0.3, f_hi=0.4),
        # the operators by themselves, as an iterative solver of one's own calls them
        dict(name="adjoint_256el_512px", kind="adjoint", n_elem=256, nx=512, ny=512, prec=mixed, f_lo=0.5),
        dict(name="adjoint_fp32_100el", kind="adjoint", n_elem=100, nx=251, ny=237, prec=fp32, f_lo=0.4),
        dict(name="forward_256el_ragged", kind="forward", n_elem=256, nx=511, ny=389, prec=mixed, f_lo=0.6),
        dict(name="forward_fp32_64el", kind="forward", n_elem=64, nx=64, ny=64, prec=fp32, f_lo=0.3),
        # ray data of a medium, as when measurements are predicted or synthesised
        dict(name="rays_256el_512px", kind="rays", n_elem=256, nx=512, ny=512, n_rays=256, n_freq=4, f_lo=0.3, f_hi=1.25),
        # tables and Green's functions for analysis outside the library
        dict(name="grid_128el_384px", kind="grid", n_elem=128, nx=384, ny=400, n_rays=256, n_freq=2, f_lo=0.4, f_hi=0.5),
        # the initial guess: three linearisations from water
        dict(name="tof_256el_256px", kind="tof", n_elem=256, nx=256, ny=256, n_rays=256, n_iter=3),
    ]


def draw(rng):
    """Another case of these ranges: rings of 64-512 elements (any size from 32 for FP32), grids of 64-512
    pixels a side, square or not, fans of 64-512 rays, one to four frequencies of 0.3-1.25 MHz."""
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["update", "update", "update", "adjoint", "forward", "rays", "grid", "tof"])
        mixed = rng.random() < 0.7
        if kind in ("update", "adjoint", "forward") and mixed:
            n = rng.choice([64, 128, 192, 256, 256, 512])
        else:
            n = int(round(math.exp(rng.uniform(math.log(32), math.log(256)))))
        nx = int(round(math.exp(rng.uniform(math.log(64), math.log(512)))))
        ny = nx if rng.random() < 0.4 else min(512, max(64, int(nx * rng.uniform(0.8, 1.25))))
        c = dict(kind=kind, n_elem=n, nx=nx, ny=ny)
        lo = round(rng.uniform(0.3, 1.0), 3)
        if kind in ("update", "adjoint", "forward"):
            c["prec"] = "bf16x3" if mixed else "fp32"
        if kind != "tof":
            c["f_lo"] = lo
        if kind in ("update", "rays", "grid"):
            c["n_freq"] = rng.randint(1, 4)
            c["f_hi"] = round(lo + rng.uniform(0.05, 0.25), 3) if c["n_freq"] > 1 else lo
        if kind in ("update", "rays", "grid", "tof"):
            c["n_rays"] = int(round(math.exp(rng.uniform(math.log(64), math.log(512)))))
        if kind == "tof":
            c["n_iter"] = rng.randint(1, 3)
        if _cost(c) <= most:
            return c


def _cost(c):
    """A case's work in operations, the FP32 contractions (which have no tensor cores) counted as more."""
    w = work(c)
    return max(w["bytes"] * 50, w["flops"] * (16 if c.get("prec") == "fp32" else 1))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _pitch(c):
    return 2.0 * 1.05 * RADIUS / (min(c["nx"], c["ny"]) - 1)


def _geom(c):
    return rb.geometry(c["n_elem"], RADIUS, c["nx"], c["ny"], _pitch(c), c.get("n_rays", 256), c_ref=C_WATER, f_ref=F_REF,
                       power_y=POWER_Y)


def _freqs(c):
    n = c.get("n_freq", 1)
    hi = c.get("f_hi", c["f_lo"])
    return [1e6 * (c["f_lo"] + (hi - c["f_lo"]) * k / max(1, n - 1)) for k in range(n)]


def _prec(c):
    return rb.RB_PREC_BF16X3 if c["prec"] == "bf16x3" else rb.RB_PREC_FP32


def _axes(c):
    h = _pitch(c)
    x = (torch.arange(c["nx"], device=DEV, dtype=torch.float64) - (c["nx"] - 1) / 2) * h
    y = (torch.arange(c["ny"], device=DEV, dtype=torch.float64) - (c["ny"] - 1) / 2) * h
    return x, y


def _elements(n):
    phi = 2 * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n
    return RADIUS * torch.cos(phi), RADIUS * torch.sin(phi)


def _support(c):
    g = _geom(c)
    r2 = math.floor((2.0 * (RADIUS - g.support_margin) / g.h) ** 2)
    jx = 2 * torch.arange(c["nx"], device=DEV) - (c["nx"] - 1)
    jy = 2 * torch.arange(c["ny"], device=DEV) - (c["ny"] - 1)
    return jy[:, None] ** 2 + jx[None, :] ** 2 <= r2


def _blur(a, sigma):
    """Gaussian smoothing of sigma pixels, the edge pixels' weights renormalised."""
    def kernel(n):
        k = torch.arange(n, device=DEV, dtype=torch.float64)
        w = torch.exp(-0.5 * ((k[:, None] - k[None, :]) / sigma) ** 2)
        return w / w.sum(1, keepdim=True)
    return kernel(a.shape[0]) @ a @ kernel(a.shape[1]).T


def _phantom(c, seed):
    """A breast in water: c_true, alpha0 and the smooth map c_init a reconstruction starts from (float32)."""
    rs = np.random.RandomState(seed % (1 << 31))
    x, y = _axes(c)
    X, Y = x[None, :], y[:, None]

    def ellipse(cx, cy, a, b, rot):
        u = (X - cx) * math.cos(rot) + (Y - cy) * math.sin(rot)
        v = -(X - cx) * math.sin(rot) + (Y - cy) * math.cos(rot)
        return (u / a) ** 2 + (v / b) ** 2 <= 1

    ct = torch.full((c["ny"], c["nx"]), C_WATER, device=DEV, dtype=torch.float64)
    a0 = torch.zeros_like(ct)
    A, B = rs.uniform(60e-3, 85e-3, 2)
    fat = ellipse(0, 0, A, B, rs.uniform(0, math.pi))
    ct[fat], a0[fat] = rs.uniform(1440, 1470), rs.uniform(0.5, 1.0)
    inner = ellipse(0, 0, 0.7 * A, 0.7 * A, 0)
    for k in range(rs.randint(8, 20)):
        r, ang = 0.7 * A * math.sqrt(rs.uniform()), rs.uniform(0, 2 * math.pi)
        big = k < 5
        a, b = rs.uniform(8e-3, 25e-3, 2) if big else rs.uniform(2e-3, 8e-3, 2)
        e = ellipse(r * math.cos(ang), r * math.sin(ang), a, b, rs.uniform(0, math.pi)) & fat & inner
        ct[e], a0[e] = rs.uniform(1500, 1560) if big else rs.uniform(1520, 1600), rs.uniform(0.5, 1.0)
    ct, a0 = _blur(ct, 2.0), _blur(a0, 2.0)
    ci = C_WATER + 0.5 * (_blur(ct, 10e-3 / _pitch(c)) - C_WATER)
    return ct.float(), a0.float(), ci.float()


def _chords(c, ct, a0, points=128):
    """Traveltime, absorption integral and length of every emitter-receiver chord through the medium."""
    n, h = c["n_elem"], _pitch(c)
    ex, ey = _elements(n)
    s = (torch.arange(points, device=DEV, dtype=torch.float64) + 0.5) / points
    T, L = (torch.empty((n, n), device=DEV, dtype=torch.float64) for _ in range(2))
    slow, att = (1.0 / ct.double()).reshape(-1), a0.double().reshape(-1)
    D = torch.hypot(ex[:, None] - ex[None, :], ey[:, None] - ey[None, :])
    for e0 in range(0, n, 64):
        px = ex[e0:e0 + 64, None, None] + (ex[None, :, None] - ex[e0:e0 + 64, None, None]) * s
        py = ey[e0:e0 + 64, None, None] + (ey[None, :, None] - ey[e0:e0 + 64, None, None]) * s
        ix = torch.clamp(torch.round(px / h + (c["nx"] - 1) / 2), 0, c["nx"] - 1).long()
        iy = torch.clamp(torch.round(py / h + (c["ny"] - 1) / 2), 0, c["ny"] - 1).long()
        at = iy * c["nx"] + ix
        T[e0:e0 + 64] = slow[at].mean(-1) * D[e0:e0 + 64]
        L[e0:e0 + 64] = att[at].mean(-1) * D[e0:e0 + 64]
    return T, L, D


def _dispersion(f):
    """Phase [cycles] per unit absorption integral of the causal power law."""
    w, wr = 2 * math.pi * f, 2 * math.pi * F_REF
    diff = wr ** (POWER_Y - 1) * math.expm1((POWER_Y - 1) * math.log(w / wr))
    return w * math.tan(0.5 * math.pi * POWER_Y) * diff * K_A * (2 * math.pi * 1e6) ** (-POWER_Y) / (2 * math.pi)


def _green(f, T, L, J, speed, kappa=0):
    """The ray Green's function in 64 bits: sqrt(c / (8 pi w J)) exp(-a L) exp(i 2 pi (f T + disp L + 1/8 - kappa / 4))."""
    amp = torch.sqrt(speed / (8 * math.pi * 2 * math.pi * f * J)) * torch.exp(-K_A * (f / 1e6) ** POWER_Y * L)
    return torch.polar(amp, 2 * math.pi * torch.remainder(f * T + _dispersion(f) * L + 0.125 - 0.25 * kappa, 1.0))


def _measured(c, ct, a0, seed):
    """Measured data [n_freq][n_elem][n_elem]: the chords' Green's functions plus 1 % noise."""
    g = torch.Generator(DEV).manual_seed(seed)
    T, L, D = _chords(c, ct, a0)
    J = torch.clamp(D, min=0.25 * _pitch(c))
    p = torch.stack([_green(f, T, L, J, torch.full_like(J, C_WATER)) for f in _freqs(c)])
    noise = torch.randn(p.shape + (2,), generator=g, device=DEV, dtype=torch.float64)
    rms = p.abs().square().mean(dim=(1, 2), keepdim=True).sqrt()
    return (p + 0.01 * rms / math.sqrt(2) * torch.view_as_complex(noise)).to(torch.complex64).contiguous()


def _mask(n):
    e = torch.arange(n, device=DEV)
    d = (e[:, None] - e[None, :]).abs()
    return torch.minimum(d, n - d) >= math.ceil(n / 8)


def _waves(c, seed, count=4):
    """Smooth random maps in [-1, 1] over the grid, one set per seed."""
    rs = np.random.RandomState((seed + 77) % (1 << 31))
    x, y = _axes(c)
    out = []
    for _ in range(count):
        kx, ky = rs.uniform(-60, 60, 2)
        out.append(torch.sin(kx * x[None, :] + ky * y[:, None] + rs.uniform(0, 2 * math.pi)).reshape(-1))
    return out


def _tables(c, seed):
    """First-arrival tables of a smooth medium: rb_cell records [n_elem][npix][4] (tag, tkey, q, l)."""
    n, npix, h = c["n_elem"], c["nx"] * c["ny"], _pitch(c)
    x, y = _axes(c)
    ex, ey = _elements(n)
    wv = _waves(c, seed)
    sup = _support(c).reshape(-1)
    tab = torch.full((n, npix, 4), -1, dtype=torch.int32, device=DEV)
    ids = (torch.arange(npix, device=DEV, dtype=torch.int64) % 60000) << 8
    for t in range(n):
        d = torch.hypot(x[None, :] - ex[t], y[:, None] - ey[t]).reshape(-1)
        a = 2 * math.pi * t / n
        bend = 0.6 * (wv[0] * math.cos(a) + wv[1] * math.sin(a)) + 0.4 * wv[2]
        tres = (d * (1e-5 * bend + 4e-6 * wv[3])).float()
        q = (torch.clamp(d, min=0.1 * h) * (1 + 0.35 * bend)).float()
        kappa = ((d > 0.15) & (bend > 0.8)).to(torch.int64)       # past a caustic
        q = torch.where(kappa == 1, -q, q)
        l = (torch.clamp(d - 0.02, min=0) * (0.6 + 0.2 * bend)).float()
        bits = tres.view(torch.int32)
        key = torch.where(bits < 0, ~bits, bits | -0x80000000)
        hit = sup & ((torch.arange(npix, device=DEV) * 7 + t * 13) % 1999 != 0)   # a few uncovered pixels
        rec = torch.stack([(ids | kappa).to(torch.int32), key, q.view(torch.int32), l.view(torch.int32)], 1)
        tab[t] = torch.where(hit[:, None], rec, tab[t])
    return tab


def _operator_inputs(c, seed):
    g = torch.Generator(DEV).manual_seed(seed)
    n, npix = c["n_elem"], c["nx"] * c["ny"]
    ct = _phantom(c, seed)[0]
    R = torch.view_as_complex(torch.randn((n, n, 2), generator=g, device=DEV)) * 0.05
    W = (_mask(n) & (torch.rand((n, n), generator=g, device=DEV) >= 0.01)).to(torch.uint8).contiguous()
    wv = _waves(c, seed + 1)
    dc = 30.0 * (wv[0] * wv[1] + 0.5 * wv[2])
    m = torch.where(_support(c).reshape(-1), -2 * _pitch(c) ** 2 * dc / ct.reshape(-1).double() ** 3, torch.zeros_like(dc))
    return dict(c=ct, R=R.to(torch.complex64).contiguous(), W=W, m=m.float().contiguous())


def prepare(case, seed):
    geom = _geom(case)
    n, npix, kind = case["n_elem"], case["nx"] * case["ny"], case["kind"]
    s = dict(kind=kind, geom=geom)
    if kind in ("adjoint", "forward"):
        s.update(_operator_inputs(case, seed), tab=_tables(case, seed), f=_freqs(case)[0], prec=_prec(case))
        s["ws"] = rb.workspace(geom, 1, s["prec"], DEV)
        if kind == "adjoint":
            s["g"] = torch.empty(npix, dtype=torch.complex64, device=DEV)
            s["h"] = torch.empty(npix, dtype=torch.float32, device=DEV)
        else:
            s["d"] = torch.empty((n, n), dtype=torch.complex64, device=DEV)
        return s
    ct, a0, ci = _phantom(case, seed)
    s["a0"] = a0.contiguous()
    if kind == "update":
        s.update(freqs=_freqs(case), prec=_prec(case), c0=ci.contiguous(), c=ci.clone(), dc=torch.empty_like(ci),
                 p=_measured(case, ct, a0, seed), diag=torch.zeros(48, dtype=torch.uint8, device=DEV))
        s["ws"] = rb.workspace(geom, len(s["freqs"]), s["prec"], DEV)
    elif kind == "tof":
        s.update(c=torch.full_like(ct, C_WATER), t=_chords(case, ct, a0)[0].contiguous(), n_iter=case["n_iter"],
                 linked=torch.ones((n, n), dtype=torch.uint8, device=DEV), c0=torch.full_like(ct, C_WATER),
                 hist=torch.zeros(case["n_iter"] + 1, dtype=torch.float64, device=DEV))
    else:
        s.update(c=ct.contiguous(), freqs=_freqs(case))
        if kind == "rays":
            s["ends"] = torch.empty((n, geom.n_rays, 56), dtype=torch.uint8, device=DEV)
            s["d"] = torch.empty((len(s["freqs"]), n, n), dtype=torch.complex64, device=DEV)
            s["linked"] = torch.empty((n, n), dtype=torch.uint8, device=DEV)
        else:
            s["tab"] = torch.empty((n, npix, 4), dtype=torch.int32, device=DEV)
            s["g"] = torch.empty((len(s["freqs"]), n, npix), dtype=torch.complex64, device=DEV)
    if "ws" not in s:
        s["ws"] = rb.workspace(geom, 1, rb.RB_PREC_FP32, DEV)
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "update":
        s["c"].copy_(s["c0"])   # an update works in place: every pass starts from the same map
        rb.rb_hf_update(s["geom"], s["c"], s["a0"], s["freqs"], s["p"], s["ws"], prec=s["prec"], dc_out=s["dc"],
                        diag_out=s["diag"])
        return dict(c=s["c"], dc=s["dc"], counts=s["diag"][24:].view(torch.int32))
    if kind == "adjoint":
        rb.rb_born_adjoint(s["geom"], s["tab"], s["c"], s["f"], s["R"], s["W"], s["g"], s["ws"], s["h"], s["prec"])
        return dict(g=s["g"], h=s["h"])
    if kind == "forward":
        rb.rb_born_forward(s["geom"], s["tab"], s["c"], s["f"], s["m"], s["d"], s["ws"], s["prec"])
        return dict(d=s["d"])
    if kind == "rays":
        rb.rb_trace_rays(s["geom"], s["c"], s["a0"], s["ends"], s["ws"])
        rb.rb_ray_forward(s["geom"], s["c"], s["ends"], s["freqs"], s["d"], s["linked"])
        e = s["ends"]
        return dict(where=e.view(torch.float64)[..., :4], tube=e.view(torch.float32)[..., 8:12],
                    counts=e.view(torch.int32)[..., 12:], p=s["d"], linked=s["linked"])
    if kind == "grid":
        rb.rb_green_grid(s["geom"], s["c"], s["a0"], s["tab"], s["ws"], s["freqs"], s["g"])
        return dict(tables=s["tab"], g=s["g"])
    s["c"].copy_(s["c0"])
    rb.rb_tof_invert(s["geom"], s["c"], s["a0"], s["t"], s["linked"], s["ws"], s["n_iter"], s["hist"])
    return dict(c=s["c"], hist=s["hist"])


def work(case):
    n, npix, kind = case["n_elem"], case["nx"] * case["ny"], case["kind"]
    nf = case.get("n_freq", 1)
    pairs = n * (n + 1) / 2          # both contractions are symmetric in emitter and receiver
    if kind == "adjoint":            # 8 operations of the gradient and 2 of the Hessian diagonal per pair and pixel
        return dict(bytes=16 * n * npix + 9 * n * n + 16 * npix, flops=10 * pairs * npix)
    if kind == "forward":
        return dict(bytes=16 * n * npix + 8 * n * n + 8 * npix, flops=8 * pairs * npix)
    # a ray: 4/pi R on average in steps of half a pixel, four stages of about 70 operations each
    rays = n * case["n_rays"] * (4 / math.pi * RADIUS / (0.5 * _pitch(case))) * 300
    if kind == "update":
        return dict(bytes=16 * npix + 8 * nf * n * n, flops=rays + 18 * pairs * npix * nf + 30 * n * npix * (1 + nf))
    if kind == "rays":
        return dict(bytes=8 * npix + 56 * n * case["n_rays"] + (8 * nf + 1) * n * n, flops=rays)
    if kind == "grid":
        return dict(bytes=8 * npix + (16 + 8 * nf) * n * npix, flops=rays + 30 * n * npix * (1 + nf))
    it = case["n_iter"]
    return dict(bytes=12 * npix + 9 * n * n, flops=rays * (it + 1) * 1.1)


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _table_green(c, s, f, t0, t1):
    """G of elements t0 .. t1 - 1 from the tables, complex128 [t][pixel] (0 at holes)."""
    h = _pitch(c)
    x, y = _axes(c)
    ex, ey = _elements(c["n_elem"])
    tab = s["tab"][t0:t1]
    d = torch.hypot(x[None, None, :] - ex[t0:t1, None, None], y[None, :, None] - ey[t0:t1, None, None]).reshape(t1 - t0, -1)
    key = tab[..., 1]
    bits = torch.where(key < 0, key & 0x7FFFFFFF, ~key)
    T = d / C_WATER + bits.view(torch.float32).double()
    q, l = tab[..., 2].view(torch.float32).double(), tab[..., 3].view(torch.float32).double()
    J = torch.clamp(q.abs(), min=0.25 * h)
    g = _green(f, T, l, J, s["c"].reshape(1, -1).double(), (tab[..., 0] & 0xFF).double())
    return torch.where((tab[..., 0] == -1) & (key == -1), torch.zeros_like(g), g)


def _exact_operator(c, seed):
    s = dict(_operator_inputs(c, seed), tab=_tables(c, seed))
    f, n, npix = _freqs(c)[0], c["n_elem"], c["nx"] * c["ny"]
    w2 = (2 * math.pi * f) ** 2
    G = torch.cat([_table_green(c, s, f, t, min(n, t + 32)) for t in range(0, n, 32)])
    if c["kind"] == "forward":
        return dict(d=w2 * (G * s["m"].double()) @ G.T)
    S = torch.where(s["W"] != 0, s["R"], torch.zeros_like(s["R"])).to(torch.complex128)
    P = G.abs().square()
    return dict(g=w2 * (G.conj() * (S @ G.conj())).sum(0), h=w2 * w2 * (P * (s["W"].double() @ P)).sum(0))


def _exact_rays(c, seed):
    """The ray fans by the same RK4 steps in 64 bits, and the linked ray data."""
    ct, a0, _ = (a.double() for a in _phantom(c, seed))
    n, nr, h, nx, ny = c["n_elem"], c["n_rays"], _pitch(c), c["nx"], c["ny"]
    ix, iy = torch.arange(nx, device=DEV), torch.arange(ny, device=DEV)
    ip, im, jp, jm = (ix + 1).clamp(max=nx - 1), (ix - 1).clamp(min=0), (iy + 1).clamp(max=ny - 1), (iy - 1).clamp(min=0)
    ic, jc = ix.clamp(1, nx - 2), iy.clamp(1, ny - 2)
    dx, dy = ((ip - im) * h)[None, :], ((jp - jm) * h)[:, None]
    dxy = (ct[jp][:, ip] - ct[jm][:, ip] - ct[jp][:, im] + ct[jm][:, im]) / (dx * dy)
    F = torch.stack([ct, (ct[:, ip] - ct[:, im]) / dx, (ct[jp] - ct[jm]) / dy,
                     (ct[:, ic + 1] - 2 * ct[:, ic] + ct[:, ic - 1]) / h ** 2, dxy,
                     (ct[jc + 1] - 2 * ct[jc] + ct[jc - 1]) / h ** 2, a0], -1).reshape(-1, 7)

    def sample(px, py, fields=F):
        u, v = (px / h + (nx - 1) / 2).clamp(0, nx - 1), (py / h + (ny - 1) / 2).clamp(0, ny - 1)
        i, j = u.floor().clamp(max=nx - 2), v.floor().clamp(max=ny - 2)
        fu, fv, at = (u - i)[:, None], (v - j)[:, None], (j * nx + i).long()
        return ((1 - fu) * (1 - fv) * fields[at] + fu * (1 - fv) * fields[at + 1] + (1 - fu) * fv * fields[at + nx] +
                fu * fv * fields[at + nx + 1])

    def slope(z):   # x, y, theta, T, Q, P, L
        f = sample(z[:, 0], z[:, 1])
        co, si, sp = torch.cos(z[:, 2]), torch.sin(z[:, 2]), f[:, 0]
        cnn = f[:, 3] * si ** 2 - 2 * f[:, 4] * si * co + f[:, 5] * co ** 2
        return torch.stack([co, si, (f[:, 1] * si - f[:, 2] * co) / sp, 1 / sp, sp * z[:, 5], -cnn / sp ** 2 * z[:, 4], f[:, 6]], 1)

    ex, ey = _elements(n)
    phi = (2 * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n)[:, None]
    th = phi + math.pi / 2 + (torch.arange(nr, device=DEV, dtype=torch.float64) + 0.5) * math.pi / nr
    x0, y0 = ex[:, None].expand(n, nr).reshape(-1), ey[:, None].expand(n, nr).reshape(-1)
    z = torch.zeros((n * nr, 7), device=DEV, dtype=torch.float64)
    z[:, 0], z[:, 1], z[:, 2], z[:, 5] = x0, y0, th.reshape(-1), 1 / sample(x0, y0)[:, 0]
    end, kap = z.clone(), torch.zeros(n * nr, device=DEV, dtype=torch.float64)
    live, ds, k = torch.arange(n * nr, device=DEV), h / 2, 0
    while live.numel() and k < 4 * RADIUS / ds:
        k += 1
        a = z[live]
        k1 = slope(a)
        k2 = slope(a + ds / 2 * k1)
        k3 = slope(a + ds / 2 * k2)
        b = a + ds / 6 * (k1 + 2 * k2 + 2 * k3 + slope(a + ds * k3))
        d = b[:, :2] - a[:, :2]
        qa, qb, qc = d.square().sum(1), 2 * (a[:, :2] * d).sum(1), a[:, :2].square().sum(1) - RADIUS ** 2
        lam = ((-qb + torch.sqrt((qb * qb - 4 * qa * qc).clamp(min=0))) / (2 * qa)).clamp(0, 1)
        out = b[:, :2].square().sum(1) >= RADIUS ** 2
        b = torch.where(out[:, None], a + lam[:, None] * (b - a), b)
        if k >= 2:
            kap[live] += torch.signbit(b[:, 4]) != torch.signbit(a[:, 4])
        z[live], end[live] = b, b
        live = live[~out]
    tres = (end[:, 3] - torch.hypot(end[:, 0] - x0, end[:, 1] - y0) / C_WATER).reshape(n, nr)
    E = end.reshape(n, nr, 7)
    where = torch.stack([E[..., 3], tres, E[..., 0], E[..., 1]], -1)
    # first arrival over the ray intervals that bracket each receiver
    ang = torch.remainder(torch.atan2(E[..., 1], E[..., 0]) - phi, 2 * math.pi)
    a, b = ang[:, :-1], ang[:, 1:]
    off = 2 * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n
    chord = torch.hypot(ex - ex[0], ey - ey[0]) / C_WATER
    fr = _freqs(c)
    p = torch.zeros((len(fr), n, n), device=DEV, dtype=torch.complex128)
    cr = sample(ex, ey, ct.reshape(-1, 1))[:, 0]
    kap = kap.reshape(n, nr)
    for dr in range(n):
        hit = (off[dr] >= torch.minimum(a, b)) & (off[dr] <= torch.maximum(a, b)) & ((b - a).abs() <= math.pi)
        lam = torch.where(b != a, (off[dr] - a) / (b - a), torch.zeros_like(a))
        T = torch.where(hit, chord[dr] + (1 - lam) * tres[:, :-1] + lam * tres[:, 1:], torch.full_like(a, math.inf))
        T, i = T.min(1, keepdim=True)
        lam = lam.gather(1, i)
        mix = lambda v: ((1 - lam) * v.gather(1, i) + lam * v.gather(1, i + 1))[:, 0]  # noqa: E731
        q, L = mix(E[..., 4]), mix(E[..., 6])
        kp = torch.where(lam <= 0.5, kap.gather(1, i), kap.gather(1, i + 1))[:, 0]
        r = (torch.arange(n, device=DEV) + dr) % n
        ok = torch.isfinite(T[:, 0])
        for w, f in enumerate(fr):
            g = _green(f, torch.where(ok, T[:, 0], 0.0), L, q.abs().clamp(min=0.25 * h), cr[r], kp)
            p[w, torch.arange(n, device=DEV), r] = torch.where(ok, g, torch.zeros_like(g))
    return dict(where=where, tube=torch.stack([E[..., 2], E[..., 4], E[..., 5], E[..., 6]], -1), counts=None, p=p, linked=None)


def exact(case, seed):
    """What run() returns in 64 bits, without the library; None for the whole calls (a full solve in 64 bits)."""
    if case["kind"] in ("adjoint", "forward"):
        return _exact_operator(case, seed)
    if case["kind"] == "rays":
        return _exact_rays(case, seed)
    return None
