"""What one sliced translation loses, against the CUDA cores' (m2l_mode 1) on the same operators.

Entries of states and operators span decades, most of all between boxes of a touching shell, so a
fixed-point slice is as precise as FP32 or FP64 only after both have been evened out.
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


def _rel(a, b):
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("case", ["sphere2", "sphere8", "adaptive"])
def test_fp64_slices(case):
    """A stage's error is at most 3e-15 of its result (the FP64 cores': 1e-15), and some six stages follow
    one another whose errors add in squares: 7.4e-15, bounded by 1e-14."""
    import torch
    from paper_1311_4257_gb300 import Plan
    if case == "adaptive":
        p, K, leaf = workloads.clustered(8.0, 3, 6000, n_clusters=3, spread=0.08), 8.0, 16
    else:
        K, leaf = float(case[6:]), 64
        p = workloads.sphere(K, 3)
    a, b = Plan(p, K, 1e-8, leaf_max=leaf), Plan(p, K, 1e-8, leaf_max=leaf, m2l_mode=1)
    for nrhs in (1, 4):
        f = torch.as_tensor(workloads.densities(p.shape[0], nrhs, nrhs), device="cuda").to(a.dtype)
        assert _rel(a.apply(f), b.apply(f)) < 1e-14


@pytest.mark.parametrize("off", [(2, 0, 0), (0, 2, 1), (-2, 0, 1), (2, 2, -2), (3, 0, 2)])
def test_fp32_slices_between_two_boxes(off):
    """Sources in one box of half a wavelength, targets in another, through one M2L: the sliced product is
    further from the FP64 one neither than the FP32 cores' (a chain of 164 FP32 multiply-adds: 3e-7 and
    more, the slices: 1e-7 or less; P2M and L2P add the same to both)."""
    import torch
    from paper_1311_4257_gb300 import Plan
    rng = np.random.default_rng(5)
    # boxes of different parents (of a whole wavelength): an odd offset of 1 crosses between two of them
    lo = np.array([{-2: 0.5, 0: -1.0, 1: -0.5, 2: -1.0, 3: -1.0}[o] for o in off])
    src = lo + 0.5 * rng.random((60, 3))
    tgt = lo + 0.5 * np.array(off) + 0.5 * rng.random((60, 3))
    p = np.concatenate([src, tgt])
    assert np.abs(p).max() <= 1.0
    f = workloads.densities(120, 16, 9)
    f[:, 60:] = 0.0
    plans = [Plan(p, 2.0, 1e-6), Plan(p, 2.0, 1e-6, m2l_mode=1), Plan(p, 2.0, 1e-6, arith=64, m2l_mode=1)]
    assert plans[0].stats()["v_pairs"] == 2
    u = [g.apply(torch.as_tensor(f, device="cuda").to(torch.complex64).to(g.dtype))[:, 60:].to(torch.complex128)
         for g in plans]
    assert _rel(u[0], u[2]) <= _rel(u[1], u[2])
