"""Plans and applies that fit the device without the sliced operator images fit with them: the images are the
last thing a plan takes, and they are given back when something else needs the memory.
"""
import gc

import pytest

import workloads

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1311_4257_gb300 import build
    build.build()


def _rel(a, b):
    return float((a - b).norm() / b.norm())


@pytest.fixture
def nearly_full():
    """fill(room): takes the device's free memory but for `room` bytes."""
    import torch
    held = []

    def fill(room):
        gc.collect()
        torch.cuda.empty_cache()
        torch.cuda.synchronize()
        free, _ = torch.cuda.mem_get_info()
        if free > room:
            held.append(torch.empty(free - room, dtype=torch.uint8, device="cuda"))

    fill.held = held
    yield fill
    held.clear()
    torch.cuda.empty_cache()


def test_images_leave_room_for_what_fitted_without_them(nearly_full):
    """Room for the plan, the batches its operators are formed in (768 MB) and half a gigabyte more: less
    than the images would take beside them."""
    import torch
    from paper_1311_4257_gb300 import Plan
    p = workloads.sphere(4.0, 5)
    plain = Plan(p, 4.0, 1e-8, m2l_mode=1)
    need = plain.plan_bytes()
    f = torch.as_tensor(workloads.densities(p.shape[0], 64, 1), device="cuda").to(plain.dtype)
    want = plain.apply(f)
    plain.close()
    u = torch.empty_like(f)
    nearly_full(need + 768 * MB + 512 * MB)
    g = Plan(p, 4.0, 1e-8)
    assert _rel(g.apply(f[:1], u[:1]), want[:1]) < 1e-12
    assert _rel(g.apply(f, u), want) < 1e-12   # the largest workspace
    g.validate()


def test_images_are_given_back_and_graphs_keep_theirs(nearly_full):
    """An allocation that the device has room for only without a plan's images takes their place, and the
    plan's applies run on; the images of a plan with a captured apply stay."""
    import torch
    from paper_1311_4257_gb300 import Plan, Server
    p = workloads.sphere(4.0, 5)
    a, b = Plan(p, 4.0, 1e-8), Plan(p, 4.0, 1e-8)
    f = torch.as_tensor(workloads.densities(p.shape[0], 1, 1), device="cuda").to(a.dtype)
    u, w, t = torch.empty_like(f), torch.empty_like(f), torch.empty_like(f)
    gr = b.graph(f, w)
    gr.launch()
    want = a.apply(f, u).clone()
    assert _rel(w, want) < 1e-13
    with_images, kept = a.plan_bytes(), b.plan_bytes()
    torch.cuda.synchronize()
    nearly_full(128 * MB)
    srv = Server(streams=1, budget_bytes=512 * MB)
    assert a.plan_bytes() < with_images - 256 * MB and b.plan_bytes() == kept
    assert _rel(a.apply(f, t), want) < 1e-12
    w.zero_()
    gr.launch()
    assert _rel(w, want) < 1e-13
    torch.cuda.synchronize()
    srv.close()


def test_apply_fails_again_after_a_workspace_that_did_not_fit(nearly_full):
    """A workspace that the device has no room for is not there for the next call either: every such call
    reports it, and smaller ones and later ones run."""
    import torch
    from paper_1311_4257_gb300 import Plan, dfmm
    p = workloads.sphere(4.0, 5)
    g = Plan(p, 4.0, 1e-5)
    f = torch.as_tensor(workloads.densities(p.shape[0], 64, 1), device="cuda").to(g.dtype)
    u = torch.empty_like(f)
    want = g.apply(f).clone()
    assert _rel(g.apply(f[:1], u[:1]), want[:1]) < 1e-6   # and everything the comparison needs is loaded
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    nearly_full(g.workspace_bytes(64) // 2)
    for _ in range(3):
        with pytest.raises(dfmm.DfmmError) as e:
            g.apply(f, u, stream=s)
        assert e.value.code == dfmm.ERR_OOM
    assert g.sync_status(s) == dfmm.OK
    g.validate()
    g.apply(f[:1], u[:1], stream=s)
    s.synchronize()
    assert _rel(u[:1], want[:1]) < 1e-6


def test_host_apply_fails_again_without_room_for_its_staging(nearly_full):
    """Room for the workspace and one of the two staging buffers of a host apply: it reports that every time,
    and runs once there is more."""
    import numpy as np
    import torch
    from paper_1311_4257_gb300 import Plan, dfmm
    p = workloads.sphere(16.0, 5)   # 64 right-hand sides: 41 MB a staging buffer
    g = Plan(p, 16.0, 1e-4)
    f = np.ascontiguousarray(workloads.densities(p.shape[0], 64, 1), dtype=np.complex64)
    fd = torch.as_tensor(f, device="cuda")
    want = g.apply(fd)
    assert _rel(g.apply(fd), want) < 1e-6
    torch.cuda.synchronize()
    one = f.nbytes
    nearly_full(one + one // 2)
    for _ in range(3):
        with pytest.raises(dfmm.DfmmError) as e:
            g.apply_host(f)
        assert e.value.code == dfmm.ERR_OOM
    nearly_full.held.clear()
    torch.cuda.empty_cache()
    assert _rel(torch.as_tensor(g.apply_host(f), device="cuda"), want) < 1e-6


def test_batch_fits_where_its_least_workspaces_do(nearly_full):
    """Room for the least workspace of every plan of a batch, with the first ones' full layouts taken first."""
    import torch
    from paper_1311_4257_gb300 import Batch, Plan
    p, nrhs = workloads.sphere(8.0, 5), 32
    plans = [Plan(p, 8.0, 1e-6) for _ in range(2)]
    fs = [torch.as_tensor(workloads.densities(p.shape[0], nrhs, k), device="cuda").to(torch.complex64) for k in range(2)]
    want = [g.apply(f) for g, f in zip(plans, fs)]
    us = [torch.empty_like(f) for f in fs]
    for w, f in zip(want, fs):
        assert _rel(w, w) == 0.0 and f.shape == w.shape
    least = plans[0].workspace_bytes(nrhs)
    torch.cuda.synchronize()
    nearly_full(2 * least + 8 * MB)
    b = Batch(plans, fs, us, graph=False, tune=False)
    b.launch()
    torch.cuda.synchronize()
    nearly_full.held.clear()
    torch.cuda.empty_cache()
    for u, w in zip(us, want):
        assert _rel(u, w) < 1e-6
    b.close()


def test_images_go_while_another_thread_applies(nearly_full):
    """Applies of two plans go on in a thread each while the main thread needs the memory of their images:
    every result is right, whether an apply ran before, on the images, or after, on the CUDA cores."""
    import threading
    import torch
    from paper_1311_4257_gb300 import Plan, Server, dfmm
    p = workloads.sphere(4.0, 5)
    plans = [Plan(p, 4.0, 1e-8) for _ in range(2)]
    f = torch.as_tensor(workloads.densities(p.shape[0], 1, 1), device="cuda").to(plans[0].dtype)
    want = plans[0].apply(f).clone()
    assert _rel(plans[1].apply(f), want) < 1e-13
    us = [[torch.zeros_like(f) for _ in range(8)] for _ in plans]
    for g, u in zip(plans, us):
        g.apply(f, u[0])
    held = sum(g.plan_bytes() for g in plans)
    torch.cuda.synchronize()
    nearly_full(64 * MB)
    stop, failed = threading.Event(), []

    def work(g, u):
        s = torch.cuda.Stream()
        try:
            k = 0
            while not stop.is_set():
                g.apply(f, u[k % 8], stream=s)
                k += 1
                s.synchronize()
        except Exception as e:   # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=work, args=a) for a in zip(plans, us)]
    for t in threads:
        t.start()
    srv = None
    for _ in range(200):   # the images are free to go between two applies
        try:
            srv = Server(streams=1, budget_bytes=256 * MB)
            break
        except dfmm.DfmmError as e:
            assert e.code == dfmm.ERR_OOM
    for _ in range(20):
        torch.cuda.synchronize()
    stop.set()
    for t in threads:
        t.join()
    assert not failed
    assert srv is not None and sum(g.plan_bytes() for g in plans) < held
    srv.close()
    nearly_full.held.clear()
    torch.cuda.empty_cache()
    for u in us:
        for v in u:
            assert _rel(v, want) < 1e-12 or not torch.any(v)
