"""A pixel that an element does not cover adds nothing to the plain FP32 forward, whatever the
perturbation holds there: a caller forms m = -2 h^2 dc / c^3 on grids whose c is 0 or undefined
outside the support.  Equal, to the bit, to m = 0 at those pixels."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_16633_gb300 import rb  # noqa: E402

R = 0.05


# one tile pair and several, one pixel chunk and many
@pytest.mark.parametrize("n,nx,ny", [(3, 9, 7), (64, 40, 41), (70, 33, 64), (150, 61, 60)])
@pytest.mark.parametrize("value", [math.nan, math.inf, -math.inf])
def test_plain_forward_ignores_m_off_the_support(n, nx, ny, value):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    g = torch.Generator(dev).manual_seed(11)
    geom = rb.geometry(n, R, nx, ny, 2.1 * R / (min(nx, ny) - 1), 16)
    npix = nx * ny
    c = 1480.0 + 40.0 * torch.rand(npix, generator=g, device=dev)
    tres = 2e-6 * torch.rand((n, npix), generator=g, device=dev)
    q = 0.005 + 0.1 * torch.rand((n, npix), generator=g, device=dev)
    l = 0.05 * torch.rand((n, npix), generator=g, device=dev)
    kap = torch.randint(0, 3, (n, npix), generator=g, device=dev, dtype=torch.int32)
    tab = torch.stack([kap, tres.view(torch.int32) | -0x80000000, q.view(torch.int32), l.view(torch.int32)], -1)
    off = torch.rand(npix, generator=g, device=dev) < 0.2     # covered by no element
    tab[:, off] = -1
    tab = tab.contiguous()
    m0 = 1e-9 * torch.randn(npix, generator=g, device=dev)
    m0[off] = 0.0
    m1 = torch.where(off, torch.full_like(m0, value), m0)
    c1 = torch.where(off, torch.full_like(c, math.nan), c)
    ws = rb.workspace(geom, 1, rb.RB_PREC_FP32, dev)
    d = [torch.full((n, n), math.nan, dtype=torch.complex64, device=dev) for _ in range(4)]
    rb.rb_born_forward(geom, tab, c, 4e5, m0, d[0], ws)
    rb.rb_born_forward(geom, tab, c1, 4e5, m1, d[1], ws)
    rb.rb_born_forward_noalloc(geom, tab, c, 4e5, m0, d[2])
    rb.rb_born_forward_noalloc(geom, tab, c1, 4e5, m1, d[3])
    assert torch.isfinite(torch.view_as_real(d[0])).all() and d[0].abs().max() > 0
    assert torch.equal(torch.view_as_real(d[1]), torch.view_as_real(d[0]))
    assert torch.equal(torch.view_as_real(d[3]), torch.view_as_real(d[2]))
