"""Row and column passes of every grid side against the FP64 oracle, at wave counts that
leave warps or CTAs of the passes partly empty (1, 5, 21 and 37 beams).

Tolerance: 1e-5 per S-matrix depth, the bound of the S-matrix parity test (FP32 FFT
round-off grows like sqrt(log N) per step; three steps here)."""
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


@pytest.mark.parametrize("n,radius,beams", [
    (64, 0.5, 1), (64, 3.4, 37), (128, 1.0, 5), (128, 2.3, 21), (256, 0.5, 1), (256, 2.3, 21),
    (384, 1.0, 5), (384, 3.4, 37), (512, 0.5, 1), (512, 2.3, 21), (768, 1.0, 5), (1024, 1.0, 5)])
def test_s_in_of_partly_filled_passes(g, n, radius, beams):
    import torch
    cell = n * 0.05
    lam = sp.LAM_200KEV
    # one more radius for the detector side, inside the band limit
    wl = sp.random_workload(n=n, n_z=3, f=1, cell=cell, n_sites=2, w=8, seed=n + beams,
                            alpha=lam * radius / cell, beta=lam * (radius + 1) / cell, dz=1.8,
                            scan_n=2)
    ctx = g.Context(0)
    sm = g.build_smatrix_for(ctx, wl)
    assert sm.n_in == beams
    ref, _ = lin.build_s_in(wl)
    out = torch.empty((sm.n_in, n // 2, n // 2), dtype=torch.complex64, device="cuda")
    for depth in range(wl.n_z):
        sm.copy_depth(depth, out)
        got = out.cpu().numpy().astype(np.complex128) / n
        err = np.linalg.norm(got - ref[depth]) / np.linalg.norm(ref[depth])
        assert err < 1e-5, (depth, err)
    # the backward (adjoint) passes and the column pass with the detector sum
    want = lin.linear_map(wl)
    assert want.max() > 0
    for got in (g.inelastic_map_for(ctx, sm, wl, "fp32"),
                g.quadratic_reference_map_for(ctx, wl)[0]):
        assert np.linalg.norm(got - want) / np.linalg.norm(want) < 1e-4
