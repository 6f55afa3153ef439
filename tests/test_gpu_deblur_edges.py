"""Deblurring filters at the edges of the solve kernel's layout against the
FP64 oracle: filters of one panel and of several with one column left, windows
larger and smaller than the image, node spacings from the smallest to the
largest the call takes (three, two and one CTA per SM). The filters are FP64
sums and factors rounded once to FP32 (6e-8); the image is an FP32 sum of up
to 121 taps and four blocks, at most 125 roundings of 6e-8 of the sum of
magnitudes: 1e-5 bounds both."""
import numpy as np
import pytest

import lsrtm_inputs as li
from oracle import deblur as db

from .test_gpu_deblur import _gpu, _handle, rel

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")


@pytest.mark.parametrize("nz,nx,s,flen,eps", [
    (9, 31, 2, 1, 1e-3),       # one tap, nodes on every second pixel
    (45, 38, 7, 3, 1e-2),      # nine columns: a panel and one column
    (30, 71, 15, 9, 3e-3),     # 81 columns, window of the image's height
    (26, 150, 48, 11, 1e-3),   # the largest spacing, image lower than a window
    (110, 55, 48, 11, 1e-3),   # the largest patch (one CTA per SM)
    (25, 33, 20, 7, 1e-3),     # one node row; sums of one lag at a time on some dx
    (64, 90, 12, 11, 1e-2),
])
def test_filters_and_image(nz, nx, s, flen, eps):
    m, r = li.image_pair(nz, nx, seed=3 * nz + nx, nrefl=6)
    m = m.astype(np.float32).astype(np.float64)
    r = r.astype(np.float32).astype(np.float64)
    h = _handle(nz, nx)
    out, F = _gpu(h, m, r, s, flen, eps)
    h.close()
    ref, Fr = db.deblur(m, r, s, flen, eps)
    assert rel(F, Fr) < 1e-5 and rel(out, ref) < 1e-5
