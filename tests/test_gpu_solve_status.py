"""A solve whose matvecs cannot complete reports it, whichever of them it was.

The plan option wait_test makes every tensor-core stage give up a bounded wait (0.2 s) on a barrier that
nothing arrives at; the status word that an apply leaves is cleared by the next one.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_4257_gb300 import build
    build.build()


@pytest.mark.parametrize("maxit", [1, 3])
def test_solve_reports_a_wait_that_gave_up(maxit):
    import torch
    from paper_1311_4257_gb300 import dfmm
    p = workloads.sphere(4.0, 31)
    b = torch.as_tensor(workloads.densities(p.shape[0], 1, 31)[0], device="cuda").to(torch.complex64)
    beta = (1.0 / workloads.POINTS_PER_SQ_WAVELENGTH) / (4.0 * np.pi)
    stalled = dfmm.Plan(p, 4.0, 1e-5, m2l_mode=2, wait_test=1)
    with pytest.raises(dfmm.DfmmError) as e:
        stalled.solve(b, 0.5, beta, maxit=maxit, tol=1e-5)
    assert e.value.code == dfmm.ERR_TIMEOUT and "gave up" in str(e.value)
    # device and stream afterwards: an ordinary plan solves the system
    x, it, rr = dfmm.Plan(p, 4.0, 1e-5).solve(b, 0.5, beta, tol=1e-5)
    assert rr <= 3e-5 and it > 1
