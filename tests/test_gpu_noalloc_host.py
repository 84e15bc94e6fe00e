"""The host side of the allocation-free apply builds every stage's work tiles once: the sizes of its layouts
come from counting them."""
import ctypes
import time

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


def _best(fn, n=20):
    t = []
    for _ in range(n):
        a = time.perf_counter()
        fn()
        t.append(time.perf_counter() - a)
    return min(t)


@pytest.mark.parametrize("eps", [1e-5, 1e-6])
def test_sizes_are_counted(eps):
    """A layout's size takes a small part of the host time of an apply that lays it out (a tenth; building
    and sorting its tiles is the most of it)."""
    import torch
    from paper_1311_4257_gb300 import Plan, lib
    L = lib()
    L.dfmm_apply_noalloc.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    p = workloads.sphere(8.0, 0)
    g = Plan(p, 8.0, eps)
    f = torch.as_tensor(workloads.densities(p.shape[0], 4, 8), device="cuda").to(g.dtype)
    u = torch.empty_like(f)
    s = torch.cuda.current_stream().cuda_stream

    def run():
        assert L.dfmm_apply_noalloc(g._h, f.data_ptr(), u.data_ptr(), 4, s) == 0

    size = _best(lambda: g.workspace_bytes(4))
    torch.cuda.synchronize()
    whole = _best(run)
    torch.cuda.synchronize()
    assert size < 0.1 * whole, (size, whole)
    assert float((u - g.apply(f)).norm() / u.norm()) < 1e-6


@pytest.mark.parametrize("nrhs", [1, 3, 64])
def test_least_workspace_is_the_cuda_cores(nrhs):
    """A plan with sliced operators runs in the workspace of one without (X lists on several levels, whose
    projection the FP64 slices take in two halves), and gives the same potentials there."""
    import torch
    from paper_1311_4257_gb300 import Plan, lib
    L = lib()
    L.dfmm_apply_noalloc.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    p = workloads.clustered(8.0, 3, 6000, n_clusters=3, spread=0.08)
    a, b = Plan(p, 8.0, 1e-8, leaf_max=16), Plan(p, 8.0, 1e-8, leaf_max=16, m2l_mode=1)
    assert a.stats()["x_pairs"] > 0
    assert a.workspace_bytes(nrhs) == b.workspace_bytes(nrhs)
    f = torch.as_tensor(workloads.densities(p.shape[0], nrhs, 8), device="cuda").to(a.dtype)
    u = torch.empty_like(f)
    s = torch.cuda.current_stream().cuda_stream
    L.dfmm_noalloc_capacity.restype = ctypes.c_int64
    rc = L.dfmm_apply_noalloc(a._h, f.data_ptr(), u.data_ptr(), nrhs, s)
    assert (rc == 0) == (b.workspace_bytes(nrhs) <= L.dfmm_noalloc_capacity())
    if rc == 0:
        assert float((u - b.apply(f)).norm() / u.norm()) < 1e-13
