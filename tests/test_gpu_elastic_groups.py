"""The cut pass of the elastic images at probe counts around its group sizes (4, 8, 16 probes
of a scan row per CTA), beam counts around its staged chunk of 32, cuts that wrap around the
cell edge and scan steps of several pixels.

Tolerance: 1e-4 against the FP64 oracle, as the elastic parity tests."""
import numpy as np
import pytest

import specimen as sp
from oracle import elastic as el
from oracle import multislice as ms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,f,radius,nsx,nsy,step", [
    (64, 1, 3.2, 1, 2, 0.37), (128, 2, 0.5, 4, 1, 0.21), (128, 2, 3.2, 5, 3, 0.11),
    (128, 4, 2.9, 9, 2, 1.30), (256, 2, 3.4, 16, 2, 0.05), (256, 4, 4.2, 17, 2, 0.83),
    (192 * 2, 3, 1.0, 24, 1, 0.29)])
def test_probe_groups(n, f, radius, nsx, nsy, step):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1908_07628_gb300 import build
    build.build()
    import paper_1908_07628_gb300 as g
    cell, lam = n * 0.1, sp.LAM_200KEV
    wl = sp.random_workload(n=n, n_z=2, f=f, cell=cell, n_sites=2, w=8, seed=n + nsx,
                            alpha=lam * f * radius / cell, beta=0.03, dz=1.8, vscale=3000.0)
    # positions from near the upper cell edge on, so that cuts wrap
    wl = wl.with_scan((nsx, nsy, 0.93 * cell + 0.013, 0.97 * cell + 0.017, step, 0.43))
    edge = lam * n / (4 * cell)
    dets = [(0.0, 0.03), (0.6 * edge, 0.0)]
    want = el.linear_images(wl, dets)
    ctx = g.Context(0)
    ctx.set_exit_plane(True)
    got = ctx.elastic_images(g.build_smatrix_for(ctx, wl), wl.scan, dets)
    for d in range(len(dets)):
        assert want[d].max() > 0
        assert ms.relative_error(want[d], got[d]) < 1e-4, d
