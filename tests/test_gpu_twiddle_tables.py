"""Twiddle tables when several host threads ask for them for the first time at once: contexts
of their own on non-blocking streams, and the contexts of one map server, which share the
server's tables.  A table read before its upload has ended gives wrong waves.

Tolerance: S-matrices have the same bits as a build with nothing else running; served maps
differ from the direct ones by the order of the FP64 map sums only (1e-12)."""
import threading

import numpy as np
import pytest

import specimen as sp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1908_07628_gb300 import build
    build.build()
    import paper_1908_07628_gb300 as pkg
    return pkg


def _workload(n):
    return sp.random_workload(n=n, n_z=2, f=2, cell=n * 0.05, n_sites=5, w=8, seed=n, scan_n=3,
                              alpha=0.02, beta=0.03, dz=1.8)


def _depths(g, ctx, wl, stream):
    import torch
    with torch.cuda.stream(stream):
        sm = g.build_smatrix_for(ctx, wl)
        out = torch.empty((wl.n_z, sm.n_in, wl.n // 2, wl.n // 2), dtype=torch.complex64,
                          device="cuda")
        for depth in range(wl.n_z):
            sm.copy_depth(depth, out[depth])
        stream.synchronize()
        sm.free()
        return out.cpu().numpy()


@pytest.mark.parametrize("n", [128, 512])
def test_fresh_contexts_at_once(g, n):
    import torch
    wl = _workload(n)
    want = _depths(g, g.Context(0), wl, torch.cuda.Stream())
    assert np.abs(want).max() > 0
    k = 6
    ready, got = threading.Barrier(k), [None] * k

    def work(i):
        stream, ctx = torch.cuda.Stream(), g.Context(0)
        ready.wait()
        got[i] = _depths(g, ctx, wl, stream)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(k)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(k):
        assert got[i] is not None and np.array_equal(got[i], want), i


@pytest.mark.parametrize("n", [256, 512])
def test_cold_server_requests_at_once(g, n):
    wl = _workload(n)
    ctx = g.Context(0)
    ctx.set_association("model")
    want = g.inelastic_map_for(ctx, g.build_smatrix_for(ctx, wl), wl, "tf32")
    ctx.close()
    req, keep = g.make_request(wl.vproj, wl.cell, wl.lam, wl.sigma, wl.dz, wl.f, wl.alpha, wl.H,
                               wl.site_slice, wl.win_x0, wl.win_y0, wl.site_x, wl.site_y,
                               wl.scan, wl.beta, precision="tf32")
    for _ in range(2):   # the second server makes its tables anew
        srv = g.Server(0, slots=4)
        ids = [srv.submit(req, keep, wl.n_types, wl.scan) for _ in range(6)]
        maps = [srv.wait(i, timeout=300)[0] for i in ids]
        srv.close()
        for m in maps:
            assert np.linalg.norm(m - want) <= 1e-12 * np.linalg.norm(want)
