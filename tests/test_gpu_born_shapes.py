"""The Born operators over the shapes their kernels branch on, against plain PyTorch in 64 bits.

Tables are drawn at random (any first-arrival record is a valid operand), the weights W are not
symmetric, and the grids leave partial pixel tiles and more or fewer tiles than the GPU has SMs.
Tolerances (relative L2): a split-precision product carries at most 3 x 2^-17 = 2.3e-5 relative
error, which a sum of random phases keeps and a sum of positive terms averages; FP32 sums of up to
1e5 terms in a few hundred partial sums stay below 1e-5.
"""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_16633_gb300 import rb  # noqa: E402

R, C0, K_A = 0.05, 1480.0, 11.512925464970229


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rb.load()
    return torch.device("cuda:0")


def _problem(dev, n, nx, ny, f=4.0e5, seed=7):
    """Geometry, random tables with holes, c, and G of the records in complex128 [n][npix]."""
    g = torch.Generator(dev).manual_seed(seed)
    geom = rb.geometry(n, R, nx, ny, 2.1 * R / (min(nx, ny) - 1), 16, power_y=1.0)
    npix = nx * ny
    c = C0 + 40.0 * torch.rand(npix, generator=g, device=dev)
    tres = 2e-6 * (torch.rand((n, npix), generator=g, device=dev) - 0.5)
    q = 0.005 + 0.1 * torch.rand((n, npix), generator=g, device=dev)
    l = 0.05 * torch.rand((n, npix), generator=g, device=dev)
    kap = torch.randint(0, 3, (n, npix), generator=g, device=dev, dtype=torch.int32)
    bits = tres.view(torch.int32)
    key = torch.where(bits < 0, ~bits, bits | -0x80000000)
    tab = torch.stack([kap, key, q.view(torch.int32), l.view(torch.int32)], -1)
    hole = torch.rand((n, npix), generator=g, device=dev) < 0.02
    tab[hole] = -1
    x = (torch.arange(nx, device=dev, dtype=torch.float64) - (nx - 1) / 2) * geom.h
    y = (torch.arange(ny, device=dev, dtype=torch.float64) - (ny - 1) / 2) * geom.h
    phi = 2 * math.pi * torch.arange(n, device=dev, dtype=torch.float64) / n
    px, py = x.repeat(ny), y.repeat_interleave(nx)
    w = 2 * math.pi * f
    G = torch.empty((n, npix), dtype=torch.complex128, device=dev)
    for t in range(n):
        d = torch.hypot(px - R * torch.cos(phi[t]), py - R * torch.sin(phi[t]))
        disp = -(2 / math.pi) * w * math.log(f / 1e6) * K_A / (2 * math.pi * 1e6)
        ph = w * (d / C0 + tres[t].double()) + disp * l[t].double() + math.pi / 4 - math.pi / 2 * kap[t].double()
        amp = torch.sqrt(c.double() / (8 * math.pi * w * q[t].double())) * torch.exp(-K_A * (f / 1e6) * l[t].double())
        G[t] = torch.where(hole[t], torch.zeros_like(ph), amp) * torch.exp(1j * ph)
    return geom, tab.contiguous(), c.contiguous(), G, f, g


def _rel(a, b):
    return (torch.linalg.vector_norm((a.to(b.dtype) - b)) / torch.linalg.vector_norm(b)).item()


# tensor cores: one pass with V beside U (64, 128), V over U's columns (192, 256), passes of 256
# elements (512, 768, 1024)
@pytest.mark.parametrize("n,nx,ny", [(64, 30, 31), (64, 180, 177), (128, 97, 60), (192, 151, 150), (256, 40, 33), (256, 160, 149),
                                     (512, 71, 70), (768, 33, 35), (1024, 64, 63)])
def test_tensor_core_adjoint_of_asymmetric_weights(dev, n, nx, ny):
    geom, tab, c, G, f, g = _problem(dev, n, nx, ny)
    S = torch.view_as_complex(torch.randn((n, n, 2), generator=g, device=dev)).contiguous()
    W = (torch.rand((n, n), generator=g, device=dev) < 0.7).to(torch.uint8).contiguous()
    ws = rb.workspace(geom, 1, rb.RB_PREC_BF16X3, dev)
    w2 = (2 * math.pi * f) ** 2
    Sw = S.to(torch.complex128) * W
    ref_g = w2 * (G.conj() * (Sw @ G.conj())).sum(0)
    P = G.abs().square()
    ref_h = w2 * w2 * (P * (W.double() @ P)).sum(0)
    for want_h in (True, False):   # the schedule differs without the Hessian contraction
        out = torch.full((nx * ny,), float("nan"), dtype=torch.complex64, device=dev)
        h = torch.full((nx * ny,), float("nan"), device=dev) if want_h else None
        rb.rb_born_adjoint(geom, tab, c, f, S, W, out, ws, h, rb.RB_PREC_BF16X3)
        assert _rel(out, ref_g) <= 3e-5
        if want_h:
            assert _rel(h, ref_h) <= 2e-5


# plain FP32: blocks of 32 elements (odd rings, the largest), one and several pixel tiles
@pytest.mark.parametrize("n,nx,ny", [(2, 20, 21), (31, 40, 37), (33, 64, 65), (100, 50, 51), (150, 61, 60), (512, 30, 33)])
def test_plain_adjoint_of_asymmetric_weights(dev, n, nx, ny):
    geom, tab, c, G, f, g = _problem(dev, n, nx, ny)
    S = torch.view_as_complex(torch.randn((n, n, 2), generator=g, device=dev)).contiguous()
    W = (torch.rand((n, n), generator=g, device=dev) < 0.7).to(torch.uint8).contiguous()
    W[0, 1] = 1
    ws = rb.workspace(geom, 1, rb.RB_PREC_FP32, dev)
    w2 = (2 * math.pi * f) ** 2
    Sw = S.to(torch.complex128) * W
    P = G.abs().square()
    out = torch.full((nx * ny,), float("nan"), dtype=torch.complex64, device=dev)
    h = torch.full((nx * ny,), float("nan"), device=dev)
    rb.rb_born_adjoint(geom, tab, c, f, S, W, out, ws, h, rb.RB_PREC_FP32)
    assert _rel(out, w2 * (G.conj() * (Sw @ G.conj())).sum(0)) <= 1e-5
    assert _rel(h, w2 * w2 * (P * (W.double() @ P)).sum(0)) <= 1e-5


# tensor cores: one to 40 pairs of row block and column group, fewer and more slices than
# splits; plain FP32: one to 36 tile pairs, one chunk and many
@pytest.mark.parametrize("prec,n,nx,ny", [("tc", 64, 20, 21), ("tc", 64, 64, 64), ("tc", 128, 97, 60), ("tc", 192, 70, 71),
                                          ("tc", 256, 40, 33), ("tc", 256, 160, 149), ("tc", 512, 71, 70), ("tc", 768, 33, 35),
                                          ("tc", 1024, 40, 41), ("fp32", 2, 20, 21), ("fp32", 63, 64, 64), ("fp32", 65, 33, 20),
                                          ("fp32", 150, 120, 121), ("fp32", 512, 30, 33)])
def test_forward_shapes(dev, prec, n, nx, ny):
    geom, tab, c, G, f, g = _problem(dev, n, nx, ny)
    m = 1e-9 * torch.randn(nx * ny, generator=g, device=dev)
    p = rb.RB_PREC_BF16X3 if prec == "tc" else rb.RB_PREC_FP32
    ws = rb.workspace(geom, 1, p, dev)
    ref = (2 * math.pi * f) ** 2 * (G * m.double()) @ G.T
    d = torch.full((n, n), float("nan"), dtype=torch.complex64, device=dev)
    rb.rb_born_forward(geom, tab, c, f, m, d, ws, p)
    assert _rel(d, ref) <= (3e-5 if prec == "tc" else 1e-5)
    if prec == "fp32":   # the same without a workspace: G synthesised per tile pair
        d.fill_(float("nan"))
        rb.rb_born_forward_noalloc(geom, tab, c, f, m, d)
        assert _rel(d, ref) <= 1e-5
