"""Pixel chunks of the plain FP32 forward: an accumulator's run of pixels is at most 2048 long, or a
128th of the grid above 512 x 512 pixels, so that its rounding does not grow with the ring."""
import pytest

from paper_2511_16633_gb300 import rb


@pytest.mark.parametrize("n_elem", [2, 63, 64, 65, 150, 256, 384, 512, 768, 1024])
def test_runs_stay_short(n_elem):
    fn = rb.load()._Z17rb_fwd_chunks_forii
    for npix in (9, 31, 32, 33, 64 * 64, 2049, 260 * 243, 300 * 300, 511 * 389, 512 * 512, 513 * 512, 1024 * 1024, 4096 * 4096):
        chunks = fn(n_elem, npix)
        assert 1 <= chunks <= 65535                       # the grid's second dimension
        assert -(-npix // chunks) <= max(2048, -(-npix // 128)), (npix, chunks)
