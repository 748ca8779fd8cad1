"""The CUDA-core contraction at the edges of its tiles: column counts (types x probe beams),
detector beams, window pixels and probes just below, at and above multiples of the tile
sides and of the K step, few and many sites (small and large tiles), shared and per-site H.

Tolerance: 1e-4 against the FP64 oracle, the bound of the FP32 path."""
import dataclasses

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


# probe and detector radii in lattice units: 0.5 -> 1 beam, 1 -> 5, 2.3 -> 21, 3.2 -> 37,
# 5.9 -> 109, 6.5 -> 137, 8.1 -> 213
@pytest.mark.parametrize("r_in,r_out,w,types,sites,scan_n", [
    (0.5, 0.5, 1, 1, 1, 1), (0.5, 1.0, 3, 1, 2, 2), (1.0, 3.2, 4, 6, 3, 4), (2.3, 2.3, 5, 3, 2, 8),
    (3.2, 5.9, 13, 2, 4, 3), (3.2, 8.1, 16, 3, 60, 9), (5.9, 6.5, 8, 1, 90, 5),
    (6.5, 8.1, 17, 2, 40, 7)])
@pytest.mark.parametrize("shared", [False, True])
def test_tile_edges(g, r_in, r_out, w, types, sites, scan_n, shared):
    n, lam = 64, sp.LAM_200KEV
    cell = n * 0.05
    wl = sp.random_workload(n=n, n_z=2, f=1, cell=cell, n_sites=sites, w=w, seed=17 + w + sites,
                            alpha=lam * r_in / cell, beta=lam * r_out / cell, dz=1.8,
                            scan_n=scan_n, n_types=types)
    H = None
    if shared:
        wl = dataclasses.replace(wl, H=np.repeat(wl.H[:1], sites, axis=0))
        H = np.ascontiguousarray(wl.H[0])
    ctx = g.Context(0)
    sm = g.build_smatrix_for(ctx, wl)
    want = lin.linear_map(wl)
    assert want.max() > 0
    got = g.inelastic_map_for(ctx, sm, wl, "fp32", H=H)
    for m in range(types):
        assert np.linalg.norm(got[m] - want[m]) / np.linalg.norm(want[m]) < 1e-4
