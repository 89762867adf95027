"""The tracer's instance that stores vertices (every update, the gridding, the time-of-flight steps)
follows the rays of the one that writes the caller's arrays: end records and vertices to the bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_16633_gb300 import rb  # noqa: E402
from wslayout import layout, vertices  # noqa: E402


@pytest.mark.parametrize("margin_steps", [40.0, 1.5, 0.5], ids=["inside", "just inside", "at the edge"])
def test_stored_vertices_are_those_of_the_rays(margin_steps):
    """margin_steps: how far the grid reaches beyond the ring, in ray steps; below one, the
    instance clamps."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    n, R, nx, n_rays = 12, 0.05, 96, 37
    h = R / ((nx - 1) / 2 - margin_steps / 2)
    geom = rb.geometry(n, R, nx, nx, h, n_rays)
    g = torch.Generator(dev).manual_seed(4)
    x = torch.linspace(0, 6, nx, device=dev)
    c = (1500 + 60 * torch.sin(x)[:, None] * torch.cos(1.3 * x)[None, :] + 3 * torch.rand((nx, nx), generator=g, device=dev)).contiguous()
    a0 = (0.5 + 0.1 * torch.cos(x)[:, None] * torch.ones_like(x)[None, :]).contiguous()
    k = geom.max_steps + 1
    f4 = lambda: torch.empty((n, n_rays, k), device=dev)  # noqa: E731
    samples = dict(vx=f4(), vy=f4(), vt=torch.empty((n, n_rays, k), dtype=torch.float64, device=dev), vq=f4(), vl=f4(),
                   vkappa=torch.empty((n, n_rays, k), dtype=torch.int32, device=dev))
    ends = torch.zeros((n, n_rays, 56), dtype=torch.uint8, device=dev)
    rb.rb_trace_rays(geom, c, a0, ends, rb.workspace(geom, 1, rb.RB_PREC_FP32, dev), samples)
    ws = rb.workspace(geom, 1, rb.RB_PREC_FP32, dev)
    tab = torch.empty((n, nx * nx, 4), dtype=torch.int32, device=dev)
    rb.rb_green_grid(geom, c, a0, tab, ws)
    off = layout(geom)
    a = rb.decode_ends(ends)
    b = rb.decode_ends(ws[off["ends"]:off["ends"] + ends.numel()].view(n, n_rays, 56))
    for name in a.dtype.names:
        assert np.array_equal(a[name], b[name]), name
    v = vertices(ws, geom, off).permute(0, 2, 1, 3)          # [fan][ray][step]
    live = torch.arange(k, device=dev) < torch.as_tensor(a["n_vert"].astype(np.int64), device=dev)[..., None]
    got = dict(vx=(v[..., 0].double() + v[..., 1].double()).float(), vy=(v[..., 2].double() + v[..., 3].double()).float(),
               vq=v[..., 5], vl=v[..., 6], vkappa=v[..., 7].contiguous().view(torch.int32))
    for name, w in got.items():
        assert torch.equal(w[live], samples[name][live]), name
    # the stored residual T - |x - x_t| / c_ref against the sampled T, to a float's last place
    phi = 2 * np.pi * torch.arange(n, device=dev, dtype=torch.float64) / n
    d = torch.hypot(v[..., 0].double() + v[..., 1].double() - R * torch.cos(phi)[:, None, None],
                    v[..., 2].double() + v[..., 3].double() - R * torch.sin(phi)[:, None, None])
    res = samples["vt"] - d / geom.c_ref
    assert torch.allclose(v[..., 4][live].double(), res[live], rtol=2e-7, atol=1e-16 + 2.0 ** -40 * R / geom.c_ref)
