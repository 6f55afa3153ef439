"""The Wiener filter's node kernel: every pair of transform lengths and sizes
with neither, planes of very different scale, and a plane with a non-finite
pixel, against the FP64 oracle.

Tolerance: the filter divides by |A|^2 + eps mean|A|^2, so a relative rounding
error u of A comes out amplified by at most about 1 / sqrt(eps) (where |A|^2 is
eps mean|A|^2): with u = 3e-7 (two split FP32 transforms) and eps = 1e-2 3e-6 a
transform; 2e-5 leaves room for the square of B and the inverse."""
import numpy as np
import pytest

import lsrtm_inputs as li
from oracle import wiener as wf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
TOL = 2e-5


def run(m, r, s, eps=1e-2):
    from paper_2508_10405_gb300 import Lsrtm
    w = li.small_case(nz=m.shape[1], nx=m.shape[2], nt=8, order=4, npml=4, nshot=1, seed=1)
    h = Lsrtm.from_workload(w)
    out = h.deblur_wiener(torch.tensor(m, device="cuda"), torch.tensor(r, device="cuda"), s, eps)
    h.close()
    return out.double().cpu().numpy()


def images(s, scale=(1.0, 1.0)):
    rng = np.random.default_rng(100 + s)
    nz, nx = 2 * s + 3, 3 * s + 5
    m = rng.standard_normal((2, nz, nx))
    r = rng.standard_normal((2, nz, nx))
    k = np.array(scale)[:, None, None]
    return (m * k).astype(np.float32), (r * k[::-1]).astype(np.float32)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("s", list(range(2, 17)) + [18, 20, 21, 24, 25, 28, 29, 30, 32])
def test_every_block_size(s):
    m, r = images(s)
    got, ref = run(m, r, s), wf.wiener(m, r, s, 1e-2)
    for q in range(2):
        assert rel(got[q], ref[q]) < TOL


@pytest.mark.parametrize("s", [7, 11, 20])
@pytest.mark.parametrize("scale", [(1e-8, 1e8), (1e10, 1.0)])
def test_planes_of_different_scale(s, scale):
    m, r = images(s, scale)
    got, ref = run(m, r, s), wf.wiener(m, r, s, 1e-2)
    for q in range(2):
        assert rel(got[q], ref[q]) < TOL


@pytest.mark.parametrize("s", [10, 20])
def test_a_spike_beside_a_plane_wave(s):
    m, r = images(s)
    m[0] = 0.0
    m[0, s, s] = 1.0
    m[1] = np.cos(0.3 * np.arange(m.shape[2]))
    got, ref = run(m, r, s), wf.wiener(m, r, s, 1e-2)
    for q in range(2):
        assert rel(got[q], ref[q]) < TOL


@pytest.mark.parametrize("s", [11, 20])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("plane", [0, 1])
def test_a_non_finite_pixel_stays_in_its_plane(s, bad, plane):
    m, r = images(s)
    ref = wf.wiener(m, r, s, 1e-2)
    m[plane, s, s] = bad
    got = run(m, r, s)
    assert not np.isfinite(got[plane]).all()
    assert rel(got[1 - plane], ref[1 - plane]) < TOL
    m, r = images(s)
    r[plane, s, s] = bad   # a block whose m'' is not finite gives zero
    got = run(m, r, s)
    assert np.isfinite(got[plane]).all()
    assert rel(got[1 - plane], ref[1 - plane]) < TOL
