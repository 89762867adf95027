"""The kernels around the large ones where their split can go wrong: cell records at the edges of
the cell tiles, the outlier selection through all its digits."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import rbgen  # noqa: E402
from oracle import geometry as ogeom  # noqa: E402
from oracle import green as ogreen  # noqa: E402
from oracle import grid as ogrid  # noqa: E402
from oracle import rays as orays  # noqa: E402
from oracle.rays import VTH, VX, VY  # noqa: E402
from paper_2511_16633_gb300 import rb  # noqa: E402


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rb.load()
    return torch.device("cuda:0")


def _t(a, dev):
    return torch.as_tensor(np.ascontiguousarray(a), device=dev).float().contiguous()


@pytest.mark.parametrize("nx,ny,n_elem", [(65, 65, 16), (66, 66, 24), (64, 67, 257), (98, 73, 8)])
def test_rays_at_cell_tile_edges(dev, nx, ny, n_elem):
    """Cells a multiple of the 32 x 8 tile, one over and one short, elements past one CTA: ray
    ends within the tracer's 1e-6 of the oracle's where they cross the ring at an angle."""
    cfg = rbgen.tiny(nx=nx, ny=ny, n_elem=n_elem, n_rays=33)
    inp = rbgen.make_inputs(rbgen.tiny(nx=nx, ny=ny, seed=cfg.seed))
    E, nv, lost = orays.trace_endpoints(ogeom.from_config(cfg), inp.c_true, inp.alpha0)
    geom = rb.geometry_from_config(cfg)
    ws = rb.workspace(geom, 1, rb.RB_PREC_FP32, dev)
    ends = torch.zeros((geom.n_elem, geom.n_rays, 56), dtype=torch.uint8, device=dev)
    rb.rb_trace_rays(geom, _t(inp.c_true, dev), _t(inp.alpha0, dev), ends, ws)
    G = rb.decode_ends(ends)
    R = cfg.ring_radius
    sinb = np.abs(np.cos(E[..., VTH]) * E[..., VX] + np.sin(E[..., VTH]) * E[..., VY]) / R
    well = sinb >= 0.1
    assert lost.sum() == 0 and (G["n_vert"] == nv).mean() >= 0.999
    assert np.max((np.hypot(G["x"] - E[..., VX], G["y"] - E[..., VY]) / R)[well]) <= 1e-6


@pytest.mark.parametrize("frac", [1e-4, 0.01, 0.3, 0.77, 0.999])
@pytest.mark.parametrize("kind", ["spread", "ties", "equal"])
def test_outlier_selection_digits(dev, kind, frac):
    """The k largest keys (|R|^2, then the lower flat index) exactly: spread values end in the
    first digits, ties and equal values go on through the index's."""
    cfg = rbgen.tiny()
    inp = rbgen.make_inputs(cfg)
    geom = rb.geometry_from_config(cfg)
    freqs = list(cfg.freqs_hz)[:2]
    n = geom.n_elem
    c, a0 = _t(inp.c_init, dev), _t(inp.alpha0, dev)
    ws = rb.workspace(geom, 2, rb.RB_PREC_FP32, dev)

    def weights(p_obs, f):
        R = torch.empty((2, n, n), dtype=torch.complex64, device=dev)
        W = torch.empty((2, n, n), dtype=torch.uint8, device=dev)
        rb.rb_data_weights(geom, c, a0, freqs, p_obs, R, W, ws, f)
        return R.cpu().numpy().ravel(), W.cpu().numpy().ravel()

    p, kept = weights(torch.zeros((2, n, n), dtype=torch.complex64, device=dev), 0.0)
    kept = kept == 1
    rng = np.random.default_rng(5)
    d = {"spread": rng.standard_normal(p.size), "ties": rng.integers(0, 3, p.size), "equal": np.zeros(p.size)}[kind]
    # imaginary parts cancel exactly, so |R|^2 is the rounded square of the real part
    p_obs = (p - (np.abs(p).max() * d).astype(np.float32)).astype(np.complex64)
    R, W = weights(torch.as_tensor(p_obs.reshape(2, n, n), device=dev), frac)
    assert not R.imag.any()
    m2 = (R.real * R.real).astype(np.float32)
    k = math.floor(frac * kept.sum())
    order = np.lexsort((np.arange(p.size), -m2.astype(np.float64)))
    order = order[kept[order]]
    want = kept.copy()
    want[order[:k]] = False
    assert np.array_equal(W == 1, want)


@pytest.mark.parametrize("nx,ny,n_elem,n_freq", [(65, 67, 9, 1), (64, 64, 17, 3), (71, 66, 33, 2)])
def test_green_with_tables(dev, nx, ny, n_elem, n_freq):
    """Green's functions written with the tables: the tables of the call without them, and the
    oracle's values within 1e-4 (relative L2, the plain path's bound)."""
    cfg = rbgen.tiny(nx=nx, ny=ny, n_elem=n_elem)
    inp = rbgen.make_inputs(rbgen.tiny(nx=nx, ny=ny, seed=cfg.seed))
    geom = rb.geometry_from_config(cfg)
    c, a0 = _t(inp.c_true, dev), _t(inp.alpha0, dev)
    ws = rb.workspace(geom, 1, rb.RB_PREC_FP32, dev)
    freqs = [cfg.freqs_hz[0] * (1 + 0.3 * k) for k in range(n_freq)]
    tabs = [torch.empty((n_elem, nx * ny, 4), dtype=torch.int32, device=dev) for _ in range(2)]
    g_out = torch.empty((n_freq, n_elem, nx * ny), dtype=torch.complex64, device=dev)
    rb.rb_green_grid(geom, c, a0, tabs[0], ws)
    rb.rb_green_grid(geom, c, a0, tabs[1], ws, freqs, g_out)
    assert torch.equal(tabs[0], tabs[1])
    g = ogeom.from_config(cfg)
    ot = ogrid.grid(g, inp.c_true, inp.alpha0)
    for j, f in enumerate(freqs):
        want = np.ravel(ogreen.green(g, ot, inp.c_true, f))
        got = np.ravel(g_out[j].cpu().numpy())
        assert np.linalg.norm(got - want) <= 1e-4 * np.linalg.norm(want)
