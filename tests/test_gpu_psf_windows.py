"""The PSF Hessian where its row blocking and its packed node windows can go
wrong: node spacings at and around the rows a thread owns (8, 4, 2, 1), so that
a thread's rows lie between two node rows, on one, or across one, against the
FP64 oracle (relative L2 1e-5, the bar of the other PSF-Hessian tests); and the
CG under a memory cap that leaves no room for a second array of node windows,
which must repeat the uncapped solve bit for bit."""
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


@pytest.mark.parametrize("shape,s", [((50, 70), 9), ((20, 22, 24), 6)])
def test_cg_without_room_for_a_second_array(shape, s):
    rng = np.random.default_rng(1)
    pv, pi, m = (dev(rng.standard_normal((2,) + shape)) for _ in range(3))
    h = handle(shape)
    h.psf_hessian(m, pv, pi, s)
    need = h.workspace_bytes()   # with one array of node windows
    x0, mis0 = h.psf_cg(m, pv, pi, 4, spacing=s)
    assert h.workspace_bytes() > need + 4096
    h.close()
    c = handle(shape, hbm_budget_bytes=need + 4096)
    x1, mis1 = c.psf_cg(m, pv, pi, 4, spacing=s)
    assert c.workspace_bytes() <= need + 4096
    assert torch.equal(x0, x1) and np.array_equal(mis0, mis1)
    c.close()
