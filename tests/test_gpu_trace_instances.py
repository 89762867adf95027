"""The tracer's instances (with and without vertex output, with and without index clamping inside
the grid) follow the same rays: equal records to the bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_16633_gb300 import rb  # noqa: E402


@pytest.mark.parametrize("margin_steps", [40.0, 1.5, 0.5], ids=["inside", "just inside", "at the edge"])
def test_instances_agree(margin_steps):
    """margin_steps: how far the grid reaches beyond the ring, in ray steps; below one, every
    instance clamps."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    n, R, nx, n_rays = 12, 0.05, 96, 37
    # half the grid = R + margin steps of h / 2
    h = R / ((nx - 1) / 2 - margin_steps / 2)
    geom = rb.geometry(n, R, nx, nx, h, n_rays)
    g = torch.Generator(dev).manual_seed(3)
    x = torch.linspace(0, 6, nx, device=dev)
    c = (1500 + 30 * torch.sin(x)[:, None] * torch.cos(1.3 * x)[None, :] + torch.rand((nx, nx), generator=g, device=dev)).contiguous()
    a0 = (0.5 + 0.1 * torch.cos(x)[:, None] * torch.ones_like(x)[None, :]).contiguous()
    ws = rb.workspace(geom, 1, rb.RB_PREC_FP32, dev)
    ends = [torch.zeros((n, n_rays, 56), dtype=torch.uint8, device=dev) for _ in range(2)]
    k = geom.max_steps + 1
    f4 = lambda: torch.empty((n, n_rays, k), device=dev)  # noqa: E731
    samples = dict(vx=f4(), vy=f4(), vt=torch.empty((n, n_rays, k), dtype=torch.float64, device=dev), vq=f4(), vl=f4(),
                   vkappa=torch.empty((n, n_rays, k), dtype=torch.int32, device=dev))
    rb.rb_trace_rays(geom, c, a0, ends[0], ws)
    rb.rb_trace_rays(geom, c, a0, ends[1], ws, samples)
    # the instance that stores vertices, through the gridding of the same rays: its tables hold
    # the first arrivals of these rays (finite, and hit almost everywhere)
    tab = torch.empty((n, nx * nx, 4), dtype=torch.int32, device=dev)
    rb.rb_green_grid(geom, c, a0, tab, ws)
    a, b = (rb.decode_ends(e) for e in ends)
    for name in a.dtype.names:
        assert np.array_equal(a[name], b[name]), name
    assert (a["n_vert"] > 0).all()
    t = rb.decode_tables(tab)
    assert t["hit"].sum() > 0.5 * n * np.pi * (R / h) ** 2 and np.isfinite(t["t_res"]).all()
