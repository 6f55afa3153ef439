"""Memory of a 2D wavefield slot: 2 x 10 ping-pong planes, 4 of node CPML
memories, the float2 image and the pseudo-Hessian (27 planes; windowed shots
carry 2 x 6 planes of their own model more), beside the 16-bit band stage. It
says how many shots a budget holds and which budgets are refused."""
import dataclasses

import numpy as np
import pytest

import lsrtm_inputs as li

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")


def handle(w, **kw):
    from paper_2508_10405_gb300 import Lsrtm
    return Lsrtm.from_workload(w, **kw)


def plane_bytes(w):
    nx = w.nx if w.geom.win_nx is None else int(np.max(w.geom.win_nx))
    pitch = (nx + 2 * w.npml + 31) // 32 * 32
    return 4 * pitch * (w.nz + 2 * w.npml)


@pytest.mark.parametrize("order", [4, 8])
@pytest.mark.parametrize("windows", [False, True])
@pytest.mark.parametrize("fp16", [False, True])
def test_planes_of_a_slot(order, windows, fp16):
    from paper_2508_10405_gb300 import BAND_FP16, BAND_FP32
    if windows:
        w = li.preset(5, nz=60, nx=150, nt=30, nshot=4, shot_dx=30, shot_x0=8, nrec_range=(6, 20), margin=9)
        w = dataclasses.replace(w, npml=10, order=order)
    else:
        w = li.small_case(nz=45, nx=70, nt=30, order=order, npml=6, nshot=4, seed=311)
    kw = dict(band_precision=BAND_FP16 if fp16 else BAND_FP32)
    b = []
    for n in (2, 1):   # (the tile tables follow the chunk height, which follows the batch: few bytes)
        h = handle(w, shots_per_batch=n, **kw)
        b.append(h.workspace_bytes())
        h.close()
    nx = w.nx if w.geom.win_nx is None else int(np.max(w.geom.win_nx))
    stage = 2 * 2 * (order // 2) * (w.nz + nx) * 4 if fp16 else 0
    slot = (39 if windows else 27) * plane_bytes(w) + stage
    assert abs(b[0] - b[1] - slot) < plane_bytes(w) // 2
