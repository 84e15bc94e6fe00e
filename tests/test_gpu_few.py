"""The few-column translation stages (automatic where operators serve a few columns each) against
the forms that serve the same stages with m2l_mode 2 (tensor cores, split) and an FP64 plan.

A sphere of 4 wavelengths sampled by n points has box pairs per operator from about one (n = 7)
to the rule's limits and beyond; right-hand sides move stages across them.
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


@pytest.mark.parametrize("n,K", [(7, 2.0), (40, 2.0), (60, 4.0), (301, 8.0), (1256, 2.0)])
def test_few_column_stages(n, K):
    """Ranks that are no multiple of 64 rows or 16 columns, operators with 1 to more than 8
    columns (several passes), more than 16 (several tiles), 1 to 3 right-hand sides.  FP32 against FP64 on the same skeletons:
    2e-6 as for the other FP32 forms (rounding of about six stages); the split form of eps 1e-5
    adds up to 2e-6 of its own."""
    import torch
    from paper_1311_4257_gb300 import Plan
    p = workloads.sphere(K, n, n=n)
    for eps, tol in ((1e-6, 2e-6), (1e-5, 4e-6)):
        g = Plan(p, K, eps)
        ref = Plan(p, K, eps, arith=64) if eps < 1e-5 else Plan(p, K, eps, m2l_mode=2)
        for nrhs in (1, 2, 3):
            f = torch.as_tensor(workloads.densities(n, nrhs, nrhs), device="cuda").to(torch.complex64)
            u = g.apply(f)
            r = ref.apply(f.to(ref.dtype)).to(torch.complex64)
            assert g.sync_status() == 0
            assert float((u - r).norm() / r.norm()) < tol, (eps, nrhs)
        g.validate()
