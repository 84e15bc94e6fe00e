"""The sliced tensor-core translations (automatic below eps 1e-5) against the CUDA-core
ones (m2l_mode 1) on the same operators.

The FP32 form's products are exact to 2^-27 of the largest entries and rounded once, so the
two forms differ by the CUDA cores' own FP32 rounding: sqrt(K) 2^-24 per stage of K <= 512
products, 1.4e-6, over about six stages in a row whose errors add in squares; 2e-6 bounds
it with the stages' partial cancellation.  The FP64 form differs by sqrt(K) 2^-53 per
stage, 3e-15, and the operators' bounded norms; 1e-12 leaves them a factor of 100.
"""
import ctypes

import numpy as np
import pytest

import workloads
from oracle import direct as OD

pytestmark = pytest.mark.gpu
TOL = {1e-6: 2e-6, 1e-8: 1e-12}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_4257_gb300 import build
    build.build()


def _pair(p, K, eps, **kw):
    from paper_1311_4257_gb300 import Plan
    return Plan(p, K, eps, **kw), Plan(p, K, eps, m2l_mode=1, **kw)


def _dev(f, g):
    import torch
    return torch.as_tensor(f, device="cuda").to(g.dtype)


def _rel(a, b):
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("eps", [1e-6, 1e-8])
@pytest.mark.parametrize("case", ["tiny", "sphere", "adaptive"])
def test_sliced_form_matches_cuda_cores(case, eps):
    """One box pair per tile up to full tiles, 1 to 64 right-hand sides (two pairs per tile),
    ranks that are no multiple of 16, plain-stored and added targets, X lists whose
    projection has K = 2 R (in two halves in the FP64 form)."""
    if case == "tiny":
        p, K, leaf, rhs = workloads.sphere(2.0, 3, n=301), 2.0, 64, (1, 64)
    elif case == "sphere":
        p, K, leaf, rhs = workloads.sphere(4.0, 5), 4.0, 64, (1, 5)
    else:
        p, K, leaf, rhs = workloads.clustered(8.0, 3, 6000, n_clusters=3, spread=0.08), 8.0, 16, (3, 1)
    a, b = _pair(p, K, eps, leaf_max=leaf)
    for nrhs in rhs:
        f = _dev(workloads.densities(p.shape[0], nrhs, nrhs), a)
        ua, ub = a.apply(f), b.apply(f)
        assert a.sync_status() == 0
        assert _rel(ua, ub) < TOL[eps], (nrhs, _rel(ua, ub))
    a.validate()
    t = np.arange(0, p.shape[0], 7)
    f64 = f.cpu().numpy().astype(np.complex128)
    ud = OD.direct(p, f64, t)
    ea, eb = (OD.rel_err(u.cpu().numpy()[:, t].astype(np.complex128), ud) for u in (ua, ub))
    assert ea < 1.1 * eb + TOL[eps] / 10, (ea, eb)


@pytest.mark.parametrize("eps,scale", [(1e-6, 1e-30), (1e-6, 1e30), (1e-8, 1e-290), (1e-8, 1e290)])
def test_sliced_form_scales_far_from_one(eps, scale):
    p = workloads.sphere(2.0, 4)
    a, b = _pair(p, 2.0, eps)
    f = _dev(workloads.densities(p.shape[0], 1, 4), a)
    ua, ub = a.apply(f * scale) / scale, b.apply(f * scale) / scale
    assert _rel(ua, ub) < TOL[eps]
    assert _rel(ua, a.apply(f)) < TOL[eps]


@pytest.mark.parametrize("eps", [1e-6, 1e-8])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_sliced_form_carries_nan_and_infinity(eps, bad):
    """A density that is not finite reaches the same potentials in both forms."""
    import torch
    p = workloads.sphere(4.0, 6, n=1500)
    a, b = _pair(p, 4.0, eps)
    f = _dev(workloads.densities(p.shape[0], 2, 6), a)
    f[1, 700] = bad
    ua, ub = a.apply(f), b.apply(f)
    fin_a, fin_b = (torch.isfinite(torch.view_as_real(u)).all(-1) for u in (ua, ub))
    assert torch.equal(fin_a, fin_b) and fin_a[0].all() and not fin_a[1].all()
    assert _rel(ua[0], ub[0]) < TOL[eps]


def test_allocation_free_apply_without_room_for_slices():
    """Where the static scratch holds the workspace but not the slices beside it, the stages
    run on the CUDA cores: what fitted without slices is accepted, with the same potentials."""
    import torch
    from paper_1311_4257_gb300 import Plan, lib
    L = lib()
    L.dfmm_apply_noalloc.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    L.dfmm_noalloc_capacity.restype = ctypes.c_int64
    p = workloads.sphere(8.0, 0)
    g = Plan(p, 8.0, 1e-8)
    cap = L.dfmm_noalloc_capacity()
    s = torch.cuda.current_stream().cuda_stream
    for nrhs in (1, 2, 3):
        f = _dev(workloads.densities(p.shape[0], nrhs, 8), g)
        u = torch.empty_like(f)
        rc = L.dfmm_apply_noalloc(g._h, f.data_ptr(), u.data_ptr(), nrhs, s)
        assert (rc == 0) == (g.workspace_bytes(nrhs) <= cap)
        if rc == 0:
            assert _rel(u, g.apply(f)) < TOL[1e-8]
