"""GMRES on right-hand sides far from one: the system is linear, so x scales with b as long as FP32
holds its entries.  The norms of the residuals and of the Krylov vectors are those of numbers whose
squares FP32 does not hold.
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


@pytest.mark.parametrize("scale", [2.0 ** -83, 2.0 ** -60, 2.0 ** -40, 2.0 ** 83])
def test_gmres_solution_scales_with_the_right_hand_side(scale):
    """Powers of two scale every FP32 operation but the apply's atomic sums exactly, so the two solutions
    differ by what the solve leaves: both satisfy the system to 3e-6 of b, and the operator's condition
    on this body is below 10."""
    import torch
    from paper_1311_4257_gb300 import Plan
    p = workloads.sphere(2.0, 7)
    b = torch.as_tensor(workloads.densities(p.shape[0], 1, 8)[0], device="cuda").to(torch.complex64)
    plan = Plan(p, 2.0, 1e-6)
    beta = (1.0 / workloads.POINTS_PER_SQ_WAVELENGTH) / (4.0 * np.pi)
    x, it, rr = plan.solve(b, 0.5, beta, tol=1e-6)
    xs, its, rrs = plan.solve(b * scale, 0.5, beta, tol=1e-6)
    assert abs(its - it) <= 1 and 0.0 < rrs <= 3e-6 and 0.0 < rr <= 3e-6
    d = (xs.to(torch.complex128) / scale - x).norm() / x.norm()
    assert float(d) < 6e-5
