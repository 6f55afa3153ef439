"""The 3D two-parameter PSF Hessian at each of its row blockings (1 to 8 rows a
thread by the node spacing) and both forms of the node blocks (packed pairs
and unpacked), against the FP64 oracle, with remainders of every tile."""
import numpy as np
import pytest

import lsrtm_inputs as li
from oracle import psf_hessian as ph

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# FP32 chains of at most 2 x 343 products over blocks of three interpolations:
# 700 roundings of 2^-24 that add at random, sqrt(700) x 6e-8 = 1.6e-6 of the
# norm, and the interpolations' few 1e-7
TOL = 1e-5


@pytest.mark.parametrize("shape,s,half", [((11, 9, 35), 2, 1), ((14, 10, 33), 3, 1), ((19, 13, 34), 4, 1),
                                          ((21, 11, 37), 7, 3), ((19, 18, 40), 9, 3)])
@pytest.mark.parametrize("transpose", [False, True])
def test_3d_rows_match_the_oracle(shape, s, half, transpose):
    from paper_2508_10405_gb300 import Lsrtm
    f32 = lambda a: np.asarray(a, np.float32)
    pv, pi = (f32(p) for p in li.psf_images3(*shape, s, seed=7))
    x = f32(np.random.default_rng(5).standard_normal((2,) + shape))
    w = li.small_case(ndim=3, nz=shape[0], ny=shape[1], nx=shape[2], nt=8, order=4, npml=4, nshot=1, seed=1)
    h = Lsrtm.from_workload(w)
    dev = [torch.tensor(a, device="cuda") for a in (x, pv, pi)]
    got = h.psf_hessian(*dev, s, half, transpose, 3).double().cpu().numpy()
    h.close()
    bl = ph.block_patches(pv.astype(np.float64), pi.astype(np.float64), s, half, 3)
    ref = ph.apply(bl, s, half, x.astype(np.float64), transpose=transpose)
    assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref)
