"""Deblurring filters of the smallest windows, which the solve gives fewer
threads: spacings on both sides of the rule, every filter length it takes, and
the longer ones that stay on the other form, against the FP64 oracle (bound as
in test_gpu_deblur_edges: one rounding of the filters, at most 125 of the image)."""
import numpy as np
import pytest

import lsrtm_inputs as li
from oracle import deblur as db

from .test_gpu_deblur import _gpu, _handle, rel

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")


@pytest.mark.parametrize("s", [2, 3, 6, 7])
@pytest.mark.parametrize("flen", [1, 5, 7, 9])
def test_small_windows(s, flen):
    nz, nx = 23, 45
    m, r = li.image_pair(nz, nx, seed=100 * s + flen, nrefl=6)
    m = m.astype(np.float32).astype(np.float64)
    r = r.astype(np.float32).astype(np.float64)
    h = _handle(nz, nx)
    out, F = _gpu(h, m, r, s, flen, 1e-2)
    h.close()
    ref, Fr = db.deblur(m, r, s, flen, 1e-2)
    assert rel(F, Fr) < 1e-5 and rel(out, ref) < 1e-5
