"""lsrtm_born_static returns before its kernels run: a wait that gave up on the
device is reported through the records, all NaN. The error word is set from
the host, so no kernel hangs or faults."""
import ctypes

import numpy as np
import pytest

import lsrtm_inputs as li

from .test_zz_no_alloc import _static_call

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("order,code", [(4, 1), (8, 2)])
def test_set_error_word_makes_every_record_nan_once(order, code):
    from paper_2508_10405_gb300 import load_library
    lib = load_library()
    w = li.small_case(nz=33, nx=41, nt=60, order=order, npml=6, nshot=2, seed=17)
    dm = torch.tensor(np.asarray(w.dm), dtype=torch.float32, device="cuda")
    d = [torch.zeros((w.geom.nrec_total, w.nt), dtype=torch.float32, device="cuda") for _ in range(3)]
    assert _static_call(lib, w, dm, d[0]) == 0
    assert torch.isfinite(d[0]).all() and d[0].abs().max() > 0
    hook = ctypes.CDLL(lib._name).lsrtm_test_static_error
    hook.argtypes, hook.restype = [ctypes.c_int], None
    hook(code)
    assert _static_call(lib, w, dm, d[1]) == 0
    assert torch.isnan(d[1]).all()
    # the next call starts clean
    assert _static_call(lib, w, dm, d[2]) == 0
    assert torch.equal(d[2], d[0])
