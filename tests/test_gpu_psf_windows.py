"""The PSF Hessian where its row blocking can go wrong: node spacings at and
around the rows a thread owns (8, 4, 2, 1), so that a thread's rows lie between
two node rows, on one, or across one, against the FP64 oracle (relative L2 1e-5,
the bar of the other PSF-Hessian tests)."""
import numpy as np
import pytest

import lsrtm_inputs as li
from oracle import psf_hessian as ph

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def dev(a):
    return torch.tensor(np.asarray(a, np.float32), device="cuda")


def handle(shape, **kw):
    from paper_2508_10405_gb300 import Lsrtm
    nd = len(shape)
    w = li.small_case(ndim=nd, nz=shape[0], ny=shape[1] if nd == 3 else 1, nx=shape[-1], nt=8, order=4, npml=4, nshot=1, seed=1)
    return Lsrtm.from_workload(w, **kw)


@pytest.mark.parametrize("s", [2, 3, 4, 7, 8, 9, 15, 17])
@pytest.mark.parametrize("mask", [1, 3])
def test_rows_and_node_rows(s, mask):
    nz, nx = 37, 45
    rng = np.random.default_rng(s)
    pv, pi = (rng.standard_normal((2, nz, nx)).astype(np.float32).astype(np.float64) for _ in range(2))
    x = rng.standard_normal((2, nz, nx)).astype(np.float32)
    half = min((s - 1) // 2, 4)
    bl = ph.block_patches(pv, pi if mask == 3 else None, s, half, mask)
    h = handle((nz, nx))
    for tr in (False, True):
        got = h.psf_hessian(dev(x), dev(pv), dev(pi) if mask == 3 else None, s, half, tr, mask).double().cpu().numpy()
        ref = ph.apply(bl, s, half, x.astype(np.float64), transpose=tr)
        assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref)
    h.close()
