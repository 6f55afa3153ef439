"""The autotuner stops at the first candidate whose steps the kernels did not
run (here skipped by the non-finite guard after a NaN perturbation) and keeps
the chunk height it had: times of skipped steps choose nothing."""
import numpy as np
import pytest

import lsrtm_inputs as li

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NONFINITE = 5


@pytest.mark.parametrize("case", [dict(nz=90, nx=40, order=4, npml=6), dict(nz=100, nx=50, order=8, npml=8),
                                  dict(ndim=3, nz=40, ny=14, nx=20, order=4, npml=5)])
def test_autotune_stops_where_steps_were_skipped(case):
    from paper_2508_10405_gb300 import Lsrtm, LsrtmError
    w = li.small_case(nt=80, nshot=2, seed=305, **case)
    h = Lsrtm.from_workload(w, guard_interval=4)
    dm = torch.tensor(np.asarray(w.dm), dtype=torch.float32, device="cuda")
    bad = dm.clone()
    bad[(0,) + tuple(n // 2 for n in w.shape)] = float("nan")
    h.born(bad)   # asynchronous: the guard trips, the call that synchronises next reports it
    before = h.kernel_launches()
    steps = 6
    with pytest.raises(LsrtmError) as e:
        h.autotune(steps=steps)
    assert e.value.status == NONFINITE
    assert h.kernel_launches() - before == 4 * steps   # one candidate
    assert len(h.autotune(steps=steps)["ms_per_step"]) > 1
    h.close()
