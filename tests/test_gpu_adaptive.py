"""Applies on adaptive octrees: the forms that run P2L, M2P and the near field beside the far field's
chain (a plain apply and a captured one) against the one that runs every step in turn (a profiled
apply), and P2M and L2P over several levels of different rank in one launch, with up to 17 right-hand sides (L2P
takes them 16 at a time).
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


@pytest.mark.parametrize("eps,nrhs", [(1e-4, 1), (1e-5, 3), (1e-5, 17), (1e-6, 1), (1e-6, 5), (1e-8, 1), (1e-8, 4)])
def test_beside_and_in_line(eps, nrhs):
    """Leaves on many levels, P2L on several (rows of their own per level) and M2P.  The forms differ in
    the order in which FP32 or FP64 terms are added: at most 1e-6 / 1e-13 of the result (about 500
    terms of at most its norm, rounding 6e-8 / 1.1e-16 each, adding as a random walk).  The clustered
    body's sums cancel little, so the same bound holds for an FP64 plan of the same skeletons
    plus the 2e-6 of the FP32 forms (4e-6 with the split form of eps above 1e-6)."""
    import torch
    from paper_1311_4257_gb300 import Plan
    p = workloads.clustered(4.0, 3, 3001)
    g = Plan(p, 4.0, eps, leaf_max=16)
    assert sum(1 for b in g.stats()["boxes"] if b) > 5
    f = torch.as_tensor(workloads.densities(3001, nrhs, 1), device="cuda").to(g.dtype)
    tol = 1e-13 if eps < 1e-6 else 1e-6
    u = g.apply(f)
    g.profile_start()
    v = g.apply(f)
    rec = g.profile_stop()
    assert g.sync_status() == 0
    assert rec["p2l_eval"]["launches"] > 1 and rec["m2p"]["launches"] >= 1
    assert float((u - v).norm() / v.norm()) < tol
    w = torch.empty_like(u)
    gr = g.graph(f, w)
    w.zero_()
    gr.launch()
    torch.cuda.synchronize()
    assert float((w - v).norm() / v.norm()) < tol
    if eps >= 1e-6:
        r = Plan(p, 4.0, eps, leaf_max=16, arith=64)
        ref = r.apply(f.to(r.dtype)).to(torch.complex64)
        assert float((u - ref).norm() / ref.norm()) < tol + (2e-6 if eps == 1e-6 else 4e-6)
