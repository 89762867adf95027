"""Where the library keeps its intermediate results in a workspace, for tests that look at them.

The offsets come from the library's own layout function; the order of its fields is read from the
header that declares them.
"""
import ctypes
import os
import re

from paper_2511_16633_gb300 import rb

HEADER = os.path.join(os.path.dirname(rb.__file__), "csrc", "rb_internal.cuh")


def layout(geom, n_freq=1, prec=rb.RB_PREC_FP32) -> dict:
    """Byte offset of every part of a workspace."""
    with open(HEADER) as f:
        body = re.search(r"struct WsLayout \{(.*?)\n\};", f.read(), re.S).group(1)
    names = re.findall(r"^\s*size_t (\w+);", body, re.M)
    buf = (ctypes.c_size_t * len(names))()
    fn = rb.load()._Z12rb_ws_layoutPK11rb_geometryi12rb_precisionP8WsLayout
    fn.argtypes, fn.restype = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_void_p], ctypes.c_size_t
    assert fn(ctypes.byref(geom), n_freq, prec, buf) == rb.rb_workspace_size(geom, n_freq, prec)
    off = dict(zip(names, buf))
    assert off["total"] == rb.rb_workspace_size(geom, n_freq, prec)
    return off


def part(ws, off, count, dtype):
    """count values of a torch dtype at a byte offset of a workspace tensor."""
    import torch
    size = torch.empty((), dtype=dtype).element_size()
    return ws[off:off + count * size].view(dtype)


def vertices(ws, geom, off):
    """The vertex stream [n_elem][max_steps + 1][n_rays][8]: xh, xl, yh, yl, t, q, l, kappa (its bits)."""
    import torch
    shape = (geom.n_elem, geom.max_steps + 1, geom.n_rays, 8)
    return part(ws, off["verts"], shape[0] * shape[1] * shape[2] * 8, torch.float32).view(shape)
