"""Kernels that have one form for small launches and one for large ones.

Row pass: few waves take k_row_pass_few, many k_row_pass, whose warps then go through several
waves.  The whole build is past that line; the static build runs the same beams in groups
that fit its 64 MiB, below it.  Both have the same bits, and the whole build is within 1e-5
of the FP64 oracle per depth (the bound of the S-matrix parity test).  The conventional
algorithm runs enough waves for the column pass with the detector sum to go through several.

Window gathers: a launch of few sites spreads a window over warps.  The map of the same sites
in batches below and above that line differs by the order of the FP64 map sums (1e-12)."""
import numpy as np
import pytest

import specimen as sp
from oracle import linear as lin

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


def _workload(n, radius, **kw):
    cell, lam = n * 0.05, sp.LAM_200KEV
    return sp.random_workload(n=n, n_z=2, f=1, cell=cell, seed=n, alpha=lam * radius / cell,
                              beta=lam * (radius + 0.5) / cell, dz=1.8, **kw)


@pytest.mark.parametrize("n,radius,beams", [
    (128, 20.0, 1257), (256, 10.0, 317), (384, 10.0, 317), (512, 6.8, 145), (768, 4.7, 69),
    (1024, 3.4, 37)])
def test_row_pass_forms(g, n, radius, beams):
    import torch
    wl = _workload(n, radius, n_sites=2, w=8, scan_n=2)
    sm = g.build_smatrix_for(g.Context(0), wl)
    assert sm.n_in == beams
    shape = (wl.n_z, beams, n // 2, n // 2)
    whole, parts = (torch.empty(shape, dtype=torch.complex64, device="cuda") for _ in range(2))
    for depth in range(wl.n_z):
        sm.copy_depth(depth, whole[depth])
    g.build_smatrix_static(torch.from_numpy(wl.vproj).cuda(), wl.cell, wl.lam, wl.sigma, wl.dz,
                           wl.f, wl.alpha, parts)
    assert torch.equal(torch.view_as_real(whole), torch.view_as_real(parts))
    ref, _ = lin.build_s_in(wl)
    for depth in range(wl.n_z):
        got = whole[depth].cpu().numpy().astype(np.complex128) / n
        err = np.linalg.norm(got - ref[depth]) / np.linalg.norm(ref[depth])
        assert err < 1e-5, (depth, err)


@pytest.mark.parametrize("n,scan_n,waves", [(64, 12, 3024), (256, 4, 336)])
def test_many_waves_of_the_conventional_algorithm(g, n, scan_n, waves):
    wl = _workload(n, 2.3, n_sites=10, w=8, scan_n=scan_n)
    assert scan_n ** 2 * (1 + wl.n_types * len(wl.site_x)) == waves   # f = 1: every site is seen
    want = lin.linear_map(wl)
    got = g.quadratic_reference_map_for(g.Context(0), wl)[0]
    assert np.linalg.norm(got - want) / np.linalg.norm(want) < 1e-4


@pytest.mark.parametrize("prec", ["tf32", "bf16x3"])
@pytest.mark.parametrize("w", [16, 17, 23, 32])   # 256, 289, 529 and 1024 window pixels
def test_gathers_below_and_above_the_line(g, prec, w):
    # 317 beams in, 349 or more out: 40 CTAs and more per site, the line at 16 per SM
    wl = _workload(128, 10.0, n_sites=200, w=w, scan_n=3)
    ctx = g.Context(0)
    sm = g.build_smatrix_for(ctx, wl)
    assert sm.n_in == 317
    for how in ("transition_first", "probe_first"):
        ctx.set_association(how)
        ctx.set_tile_width(128)
        ctx.set_batch_sites(0)
        many = g.inelastic_map_for(ctx, sm, wl, prec)
        ctx.set_batch_sites(5)
        few = g.inelastic_map_for(ctx, sm, wl, prec)
        assert np.linalg.norm(few - many) <= 1e-12 * np.linalg.norm(many), how
    want = g.inelastic_map_for(ctx, sm, wl, "fp32")
    assert np.linalg.norm(many - want) / np.linalg.norm(want) < 1e-3
