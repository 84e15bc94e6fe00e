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
