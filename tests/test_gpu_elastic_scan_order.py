"""Elastic images of scans that run towards smaller x, of steps that jump over several cut
widths, and of launches that leave SMs without a CTA of 16 probes.

Tolerance: 1e-4 against the FP64 oracle, as the elastic parity tests; the same scan run the
other way gives the same positions up to FP64 rounding, so its images agree to 1e-5."""
import numpy as np
import pytest

import specimen as sp
from oracle import elastic as el
from oracle import multislice as ms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,f,radius,nsx,nsy,step", [
    (128, 2, 2.3, 7, 2, -0.31), (128, 2, 2.3, 16, 1, -0.11), (128, 1, 3.4, 16, 2, -0.07),
    (256, 4, 4.2, 20, 3, -0.2), (256, 4, 4.2, 33, 1, -1.37), (256, 2, 3.4, 19, 1, 3.9),
    (64, 1, 2.3, 9, 1, 0.13), (512, 4, 4.2, 24, 2, -0.2)])
def test_scan_order(n, f, radius, nsx, nsy, step):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1908_07628_gb300 import build
    build.build()
    import paper_1908_07628_gb300 as g
    cell, lam = n * 0.1, sp.LAM_200KEV
    wl = sp.random_workload(n=n, n_z=2, f=f, cell=cell, n_sites=2, w=8, seed=n + nsx,
                            alpha=lam * f * radius / cell, beta=0.03, dz=1.8, vscale=3000.0)
    # a quarter pixel off the grid's midpoints, so that no window edge is a matter of rounding
    px = cell / (n // 2)
    x0, step = (0.3 + 0.25 / 16) * px, round(step / px * 16) * px / 16
    there = (nsx, nsy, x0, 0.97 * cell + 0.017, step, 0.43)
    back = (nsx, nsy, x0 + (nsx - 1) * step, 0.97 * cell + 0.017, -step, 0.43)
    edge = lam * n / (4 * cell)
    dets = [(0.0, 0.03), (0.6 * edge, 0.0)]
    wl = wl.with_scan(there)
    want = el.linear_images(wl, dets)
    ctx = g.Context(0)
    ctx.set_exit_plane(True)
    sm = g.build_smatrix_for(ctx, wl)
    got = ctx.elastic_images(sm, there, dets)
    other = ctx.elastic_images(sm, back, dets)
    for d in range(len(dets)):
        assert want[d].max() > 0
        assert ms.relative_error(want[d], got[d]) < 1e-4, d
        assert ms.relative_error(got[d], other[d][:, ::-1]) < 1e-5, d
