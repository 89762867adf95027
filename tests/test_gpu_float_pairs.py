"""The float-pair distance and traveltime of the Green's functions keep the accuracy of the general
pair operations (add, square, square root, product), measured against 64 bits on the same inputs:
neither their rms error nor the largest may exceed it."""
import ctypes
import math
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_16633_gb300 import _build, rb  # noqa: E402

SOURCE = r"""
#include "rb_internal.cuh"
// out [4][n]: errors of the distance (as used, general) and of the traveltime (as used, general), both
// relative to the distance
__global__ void k_errors(GeoDev G, int n, const int* ix, const int* iy, const float4* el, const float* tres, DF inv_c, double* out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const float4 e = el[k];
    const DF ex{e.x, e.y}, ey{e.z, e.w};
    const DF X = df_pixel_coord(ix[k], G.cxg, G.h_hi, G.h_lo), Y = df_pixel_coord(iy[k], G.cyg, G.h_hi, G.h_lo);
    auto val = [](DF a) { return (double)a.hi + (double)a.lo; };
    const double dx = val(X) - val(ex), dy = val(Y) - val(ey), d = sqrt(dx * dx + dy * dy);
    const DF used = pixel_elem_dist(G, ix[k], iy[k], ex, ey);
    const DF gx = df_sub(X, ex), gy = df_sub(Y, ey), g2 = df_add(df_sqr(gx), df_sqr(gy));
    const DF gen = df_sqrt(g2);
    out[k] = fabs(val(used) - d) / d;
    out[n + k] = fabs(val(gen) - d) / d;
    rb_cell rec{0u, f2key(tres[k]), 0.01f, 0.f};
    const float4 s = synth_record(rec, 38.f, gen, inv_c.hi, inv_c.lo, 1e-4f);
    const double t0 = val(gen) * val(inv_c), t = t0 + (double)tres[k];
    out[2 * n + k] = fabs(val(DF{s.x, s.y}) - t) / t0;
    out[3 * n + k] = fabs(val(df_add(df_mul(gen, inv_c), DF{tres[k], 0.f})) - t) / t0;
}
extern "C" int errors(const void* G, int n, const int* ix, const int* iy, const float4* el, const float* tres, float ch, float cl,
                      double* out) {
    k_errors<<<(n + 255) / 256, 256>>>(*(const GeoDev*)G, n, ix, iy, el, tres, DF{ch, cl}, out);
    if (cudaGetLastError() != cudaSuccess) return 1;
    return cudaDeviceSynchronize() != cudaSuccess;
}
extern "C" int geo_bytes() { return (int)sizeof(GeoDev); }
// the parts of GeoDev that the pixel coordinates use
extern "C" void fill_geo(void* p, float cxg, float cyg, double h) {
    GeoDev& G = *(GeoDev*)p;
    const DF d = df_from_double(h);
    G.cxg = cxg;
    G.cyg = cyg;
    G.h_hi = d.hi;
    G.h_lo = d.lo;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rb.load()
    d = tmp_path_factory.mktemp("pairs")
    src, so = str(d / "pairs.cu"), str(d / "pairs.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-I", _build.CSRC, "-I", os.path.join(_build.ROOT, "include"),
                    "-shared", src, "-o", so], check=True)
    lib = ctypes.CDLL(so)
    P = ctypes.c_void_p
    lib.errors.argtypes = [P, ctypes.c_int, P, P, P, P, ctypes.c_float, ctypes.c_float, P]
    lib.fill_geo.argtypes = [P, ctypes.c_float, ctypes.c_float, ctypes.c_double]
    return lib


@pytest.mark.parametrize("nx,ny,R", [(512, 512, 0.11), (511, 389, 0.11), (64, 64, 0.05), (1024, 1000, 0.1), (96, 101, 0.137)])
def test_pairs_are_as_accurate_as_the_general_operations(lib, nx, ny, R):
    dev, n = torch.device("cuda:0"), 1 << 22
    g = torch.Generator(dev).manual_seed(nx + ny)
    h = 2.1 * R / (min(nx, ny) - 1)
    ix = torch.randint(0, nx, (n,), generator=g, device=dev, dtype=torch.int32)
    iy = torch.randint(0, ny, (n,), generator=g, device=dev, dtype=torch.int32)
    phi = 2 * math.pi * torch.randint(0, 256, (n,), generator=g, device=dev).double() / 256
    el = []
    for v in (R * torch.cos(phi), R * torch.sin(phi)):
        el += [v.float(), (v - v.float().double()).float()]
    el = torch.stack(el, -1).contiguous()
    tres = (4e-6 * (torch.rand(n, generator=g, device=dev) - 0.5)).contiguous()
    inv = 1.0 / 1480.0
    ch = float(torch.tensor(inv, dtype=torch.float32))
    geo = ctypes.create_string_buffer(lib.geo_bytes())
    lib.fill_geo(geo, 0.5 * (nx - 1), 0.5 * (ny - 1), h)
    out = torch.empty((4, n), dtype=torch.float64, device=dev)
    assert lib.errors(geo, n, ix.data_ptr(), iy.data_ptr(), el.data_ptr(), tres.data_ptr(), ch, inv - ch, out.data_ptr()) == 0
    rms, top = out.square().mean(1).sqrt().tolist(), out.max(1).values.tolist()
    for k, what in ((0, "distance"), (2, "traveltime")):
        # over four million random inputs the rms is known to a thousandth; the largest of sums of
        # half a dozen roundings, to some per cent
        assert rms[k] <= 1.002 * rms[k + 1], (what, [math.log2(v) for v in rms])
        assert top[k] <= 1.1 * top[k + 1], (what, [math.log2(v) for v in top])
