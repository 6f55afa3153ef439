"""The 2D and the fused 3D time-step kernels where their blocking can go wrong, against the FP64
oracle: padded depths that end in the middle of a group of two rows, padded
widths one column around the CTA's 240 (order 8) or 248 (order 4) output
columns, absorbing strips of odd width (whose 16-bit band values are fetched
in pairs), z-chunks that start in the strips, a free surface, and aperture
windows around the CTA width; in 3D grids around the 32 x 12 tile, strips
narrower and wider than the halo, one and several z-chunks. Tolerance: the FP32 bar of the operators,
relative L2 1e-4. 16-bit bands: on grids this small the format's own error is
not bounded beforehand, but it falls with the mantissa (8 bits of BF16, 11 of
FP16: 8x), so FP16's is asked to be under a third of BF16's; values from a
wrong place of the band would leave both large."""
import dataclasses

import numpy as np
import pytest

import lsrtm_inputs as li
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("order,nz,nx,npml,fs", [
    (4, 20, 30, 5, False), (4, 9, 238, 5, False), (4, 17, 239, 5, True), (8, 21, 229, 5, False), (8, 20, 231, 5, False),
    (8, 12, 230, 9, True), (8, 130, 33, 7, False), (4, 131, 21, 11, True),
])
def test_groups_and_tiles(order, nz, nx, npml, fs):
    from paper_2508_10405_gb300 import BAND_BF16, BAND_FP16, Lsrtm
    w = li.small_case(nz=nz, nx=nx, nt=120, order=order, npml=npml, nshot=2, nrec=60, seed=nz + nx)
    if fs:   # no source on the surface row
        w = dataclasses.replace(w, free_surface=True)
    h = Lsrtm.from_workload(w)
    d = h.born(torch.tensor(w.dm, dtype=torch.float32, device="cuda"))
    ref = oracle.born(w, w.dm)
    assert rel(d.cpu(), ref) < 1e-4
    dres = np.random.default_rng(nz).standard_normal(ref.shape)
    g, ph = h.adjoint(torch.tensor(dres, dtype=torch.float32, device="cuda"), pseudo_hessian=True)
    gref = oracle.adjoint(w, dres)
    assert rel(g.cpu(), gref) < 1e-4
    assert rel(ph.cpu(), oracle.pseudo_hessian(w)) < 1e-4
    assert rel(h.model().cpu(), oracle.model(w)) < 1e-4
    h.close()
    e = {}
    for bands in (BAND_BF16, BAND_FP16):
        h = Lsrtm.from_workload(w, band_precision=bands)
        e[bands] = rel(h.adjoint(torch.tensor(dres, dtype=torch.float32, device="cuda")).cpu(), gref)
        h.close()
    assert e[BAND_FP16] < e[BAND_BF16] / 3


@pytest.mark.parametrize("order,widths", [(8, (219, 220, 221)), (4, (228, 229, 12))])
def test_windows_around_the_cta_width(order, widths):
    from paper_2508_10405_gb300 import Lsrtm
    w = li.small_case(nz=19, nx=260, nt=80, order=order, npml=10, nshot=3, seed=3)
    x0 = np.array([3, 0, 30], np.int32)
    wn = np.array(widths, np.int32)
    nx, src, ptr, idx = w.nx, [], [0], []
    for s in range(3):
        cols = x0[s] + np.array([1, wn[s] // 2, wn[s] - 1])
        src.append(nx + x0[s] + wn[s] // 2)
        idx.append(2 * nx + cols)
        ptr.append(ptr[-1] + cols.size)
    w = dataclasses.replace(w, geom=li.Geometry(np.array(src, np.int32), np.array(ptr, np.int32),
                                                np.concatenate(idx).astype(np.int32), x0, wn))
    h = Lsrtm.from_workload(w)
    d = h.born(torch.tensor(w.dm, dtype=torch.float32, device="cuda"))
    ref = oracle.born(w, w.dm)
    assert rel(d.cpu(), ref) < 1e-4
    dres = np.random.default_rng(1).standard_normal(ref.shape)
    g = h.adjoint(torch.tensor(dres, dtype=torch.float32, device="cuda"))
    assert rel(g.cpu(), oracle.adjoint(w, dres)) < 1e-4
    h.close()


@pytest.mark.parametrize("order,nz,ny,nx,npml,fs,shots", [
    (4, 9, 1, 20, 6, False, 1), (4, 20, 13, 21, 5, True, 3), (8, 10, 4, 16, 4, False, 2), (8, 33, 12, 49, 8, False, 1),
    (8, 21, 29, 17, 9, True, 2), (4, 12, 37, 61, 3, False, 2),
])
def test_3d_tiles(order, nz, ny, nx, npml, fs, shots):
    from paper_2508_10405_gb300 import BAND_BF16, BAND_FP16, Lsrtm
    w = li.small_case(ndim=3, nz=nz, ny=max(ny, 3), nx=nx, nt=60, order=order, npml=npml, nshot=shots, nrec=80, seed=nz + nx)
    if fs:
        w = dataclasses.replace(w, free_surface=True)
    h = Lsrtm.from_workload(w)
    d = h.born(torch.tensor(w.dm, dtype=torch.float32, device="cuda"))
    ref = oracle.born(w, w.dm)
    assert rel(d.cpu(), ref) < 1e-4
    dres = np.random.default_rng(nz).standard_normal(ref.shape)
    gref = oracle.adjoint(w, dres)
    assert rel(h.adjoint(torch.tensor(dres, dtype=torch.float32, device="cuda")).cpu(), gref) < 1e-4
    h.close()
    e = {}
    for bands in (BAND_BF16, BAND_FP16):
        h = Lsrtm.from_workload(w, band_precision=bands)
        e[bands] = rel(h.adjoint(torch.tensor(dres, dtype=torch.float32, device="cuda")).cpu(), gref)
        h.close()
    assert e[BAND_FP16] < e[BAND_BF16] / 3
