"""The plain FP32 operators at the sizes where their kernels change: rings below 48 elements, whose
adjoint multiplies out the full sums (one or two elements a thread, chunks of eight r), and
forwards of few pixel chunks, which a warp sums by itself.  References and tolerances as in
test_gpu_born_shapes.py (FP32 sums against 64 bits: 1e-5 relative L2)."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_16633_gb300 import rb  # noqa: E402
from test_gpu_born_shapes import _problem, _rel, dev  # noqa: E402,F401


@pytest.mark.parametrize("n,nx,ny", [(3, 9, 7), (7, 40, 37), (8, 33, 32), (9, 40, 41), (24, 50, 51), (32, 64, 63), (40, 61, 60),
                                     (47, 64, 65), (48, 64, 65), (63, 40, 40), (64, 33, 31)])
def test_adjoint_of_small_rings(dev, n, nx, ny):  # noqa: F811
    geom, tab, c, G, f, g = _problem(dev, n, nx, ny)
    S = torch.view_as_complex(torch.randn((n, n, 2), generator=g, device=dev)).contiguous()
    W = (torch.rand((n, n), generator=g, device=dev) < 0.7).to(torch.uint8).contiguous()
    W[0, 1] = 1
    ws = rb.workspace(geom, 1, rb.RB_PREC_FP32, dev)
    w2 = (2 * math.pi * f) ** 2
    Sw = S.to(torch.complex128) * W
    P = G.abs().square()
    for want_h in (True, False):
        out = torch.full((nx * ny,), float("nan"), dtype=torch.complex64, device=dev)
        h = torch.full((nx * ny,), float("nan"), device=dev) if want_h else None
        rb.rb_born_adjoint(geom, tab, c, f, S, W, out, ws, h, rb.RB_PREC_FP32)
        assert _rel(out, w2 * (G.conj() * (Sw @ G.conj())).sum(0)) <= 1e-5
        if want_h:
            assert _rel(h, w2 * w2 * (P * (W.double() @ P)).sum(0)) <= 1e-5


# two chunks (on the coarsest grid whose h / 4, the floor of |q|, lies below the tables' q), eight,
# ten, and the fixed scratch's single chunk for a thousand elements
@pytest.mark.parametrize("n,nx,ny", [(70, 7, 7), (33, 16, 16), (70, 17, 17), (600, 16, 15), (1000, 12, 11)])
def test_forward_of_few_chunks(dev, n, nx, ny):  # noqa: F811
    geom, tab, c, G, f, g = _problem(dev, n, nx, ny)
    m = 1e-9 * torch.randn(nx * ny, generator=g, device=dev)
    ref = (2 * math.pi * f) ** 2 * (G * m.double()) @ G.T
    ws = rb.workspace(geom, 1, rb.RB_PREC_FP32, dev)
    d = torch.full((n, n), float("nan"), dtype=torch.complex64, device=dev)
    rb.rb_born_forward(geom, tab, c, f, m, d, ws, rb.RB_PREC_FP32)
    assert _rel(d, ref) <= 1e-5
    d.fill_(float("nan"))
    rb.rb_born_forward_noalloc(geom, tab, c, f, m, d)
    assert _rel(d, ref) <= 1e-5
