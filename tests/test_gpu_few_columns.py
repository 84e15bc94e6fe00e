"""The few-column translation stages over their whole range of right-hand sides, with evidence that they run:
below eps 1e-5 a stage in this form has no split of its source, one in the sliced form has.
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


def _splits(g, f):
    g.apply(f)   # the profile is the workspace's: laid out for this many right-hand sides first
    g.profile_start()
    u = g.apply(f)
    rec = g.profile_stop()
    return u, rec.get("split", {"launches": 0})["launches"]


@pytest.mark.parametrize("nrhs,few", [(1, True), (4, True), (5, True), (7, True), (8, True), (11, True), (12, True),
                                      (13, False), (64, False)])
def test_two_boxes(nrhs, few):
    """One box pair per operator and nrhs columns, the rule's limit at 12: tiles of one pair with every number
    of columns per thread.  FP32 against FP64 on the same skeletons: 2e-6 as for the other FP32 forms."""
    import torch
    from paper_1311_4257_gb300 import Plan
    rng = np.random.default_rng(5)
    p = np.concatenate([-1.0 + 0.5 * rng.random((60, 3)), [0.0, -1.0, -1.0] + 0.5 * rng.random((60, 3))])
    g, ref = Plan(p, 2.0, 1e-6), Plan(p, 2.0, 1e-6, arith=64)
    assert g.stats()["v_pairs"] == 2
    f = torch.as_tensor(workloads.densities(120, nrhs, nrhs), device="cuda").to(torch.complex64)
    u, splits = _splits(g, f)
    assert (splits == 0) == few
    r = ref.apply(f.to(ref.dtype)).to(torch.complex64)
    assert float((u - r).norm() / r.norm()) < 2e-6


def test_sums_are_the_cuda_cores(nrhs=4):
    """Sources in one box, targets in another, so that each target state has one addition: the potentials are
    those of the CUDA-core stage (16 right-hand sides) to the bit."""
    import torch
    from paper_1311_4257_gb300 import Plan
    rng = np.random.default_rng(6)
    p = np.concatenate([-1.0 + 0.5 * rng.random((60, 3)), [0.0, -1.0, -0.5] + 0.5 * rng.random((60, 3))])
    g = Plan(p, 2.0, 1e-6, m2l_mode=1)
    f = torch.as_tensor(workloads.densities(120, 16, 3), device="cuda").to(torch.complex64)
    f[:, 60:] = 0.0
    many, few = g.apply(f), g.apply(f[:nrhs].contiguous())
    assert torch.equal(many[:nrhs, 60:], few[:, 60:])
    assert float(few[:, 60:].abs().min()) > 0.0


@pytest.mark.parametrize("n,K", [(301, 2.0), (700, 3.0)])
def test_bodies_with_many_right_hand_sides(n, K):
    """Several pairs per tile and columns across the limits of tiles and threads, some stages in the form and
    some not."""
    import torch
    from paper_1311_4257_gb300 import Plan
    p = workloads.sphere(K, n, n=n)
    g, ref = Plan(p, K, 1e-6), Plan(p, K, 1e-6, arith=64)
    for nrhs in (1, 4, 5, 7, 8, 12):
        f = torch.as_tensor(workloads.densities(n, nrhs, nrhs), device="cuda").to(torch.complex64)
        r = ref.apply(f.to(ref.dtype)).to(torch.complex64)
        u = g.apply(f)
        assert g.sync_status() == 0
        assert float((u - r).norm() / r.norm()) < 2e-6, nrhs
