"""The pixel sums of a time-of-flight step against the same sums in 64 bits from its own vertices and
coefficients.

The sums are whole numbers in units of the largest coefficient times the ray step over 2^40.  A
bilinear weight is formed in floats from a pixel coordinate below 128 (half an ulp, 2^-18 pixels,
and as much again from the midpoint): 2^-16 of the segment's length at most, which is the bound
relative to the largest pixel's sum of |coefficient| x length.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_16633_gb300 import rb  # noqa: E402
from wslayout import layout, part, vertices  # noqa: E402


# ray steps in pixels: the default; one that skips quads and moves diagonally; long stays in one
# quad and rays of many 64-step pieces (steps just above and below a power of two among them)
@pytest.mark.parametrize("ratio", [0.5, 1.7, 0.9, 0.02])
@pytest.mark.parametrize("nx,ny,R", [(66, 61, 0.05), (40, 44, 0.041)])
def test_deposits(ratio, nx, ny, R):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    n, n_rays = 10, 23
    h = 2.1 * R / (min(nx, ny) - 1)
    geom = rb.geometry(n, R, nx, ny, h, n_rays, ds=ratio * h)
    x, y = torch.linspace(0, 5, nx, device=dev), torch.linspace(0, 4, ny, device=dev)
    c = (1500 + 50 * torch.sin(y)[:, None] * torch.cos(1.3 * x)[None, :]).contiguous()
    a0 = torch.zeros_like(c)
    t = torch.empty((n, n), dtype=torch.float64, device=dev)
    linked = torch.empty((n, n), dtype=torch.uint8, device=dev)
    rb.rb_tof_times(geom, c, a0, t, rb.workspace(geom, 1, rb.RB_PREC_FP32, dev), linked)
    g = torch.Generator(dev).manual_seed(5)
    t = (t * (1 + 0.01 * torch.randn((n, n), generator=g, device=dev, dtype=torch.float64))).contiguous()
    ends = torch.zeros((n, n_rays, 56), dtype=torch.uint8, device=dev)
    ws = rb.workspace(geom, 1, rb.RB_PREC_FP32, dev)
    rb.rb_trace_rays(geom, c, a0, ends, ws)
    nv = rb.decode_ends(ends)["n_vert"]
    rb.rb_tof_invert(geom, c.clone(), a0, t, linked, ws, 1)
    off = layout(geom)
    al = lambda b: (b + 255) // 256 * 256  # noqa: E731
    at = off["tof"] + al(n * n * 16) + al(n * n_rays * 4)
    coef = part(ws, at, n * n_rays * 2, torch.float32).view(n, n_rays, 2).double().cpu().numpy()
    at += al(n * n_rays * 8)
    sums = [part(ws, at + k * al(nx * ny * 8), nx * ny, torch.int64).cpu().numpy() for k in range(2)]
    top = part(ws, at + 2 * al(nx * ny * 8), 2, torch.float32).double().cpu().numpy()
    assert np.array_equal(top, np.abs(coef).reshape(-1, 2).max(0)) and (top > 0).all()
    v = vertices(ws, geom, off).double().cpu().numpy()
    X, Y = v[..., 0] + v[..., 1], v[..., 2] + v[..., 3]      # [fan][step][ray]
    seg = np.arange(1, geom.max_steps + 1)[None, :, None] < nv[:, None, :]
    dx, dy = np.diff(X, axis=1)[seg], np.diff(Y, axis=1)[seg]
    l = np.hypot(dx, dy)
    u = np.clip((X[:, :-1][seg] + 0.5 * dx) / h + (nx - 1) / 2, 0, nx - 1)
    w = np.clip((Y[:, :-1][seg] + 0.5 * dy) / h + (ny - 1) / 2, 0, ny - 1)
    i, j = np.minimum(u.astype(int), nx - 2), np.minimum(w.astype(int), ny - 2)
    fu, fw = u - i, w - j
    fan, _, ray = np.nonzero(seg)
    for k in range(2):
        a = coef[fan, ray, k]
        ref, mag = np.zeros(nx * ny), np.zeros(nx * ny)
        for di, dj, wt in ((0, 0, (1 - fu) * (1 - fw)), (1, 0, fu * (1 - fw)), (0, 1, (1 - fu) * fw), (1, 1, fu * fw)):
            np.add.at(ref, (j + dj) * nx + i + di, a * wt * l)
            np.add.at(mag, (j + dj) * nx + i + di, np.abs(a) * l)
        got = sums[k].astype(np.float64) * top[k] * geom.ds / 2.0 ** 40
        assert np.abs(got - ref).max() <= 2.0 ** -16 * mag.max()
