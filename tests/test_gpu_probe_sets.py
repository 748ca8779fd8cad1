"""Probe rows shared by the sites of a map (gathered once per distinct probe set) against
the FP64 oracle and against the per-site gather: crystals whose windows hold the whole scan,
part of it, and maps where no two sites see the same probes; both groupings, both
tensor-core precisions, batches that split a slice.

Tolerance: the bounds of the precision classes (1e-4 TF32, 1e-3 BF16 hi + lo)."""
import numpy as np
import pytest

import specimen as sp
from oracle import linear as lin

pytestmark = pytest.mark.gpu

EPS = {"tf32": 1e-4, "bf16x3": 1e-3}


@pytest.mark.parametrize("kind", ["whole_scan", "partly", "distinct"])
def test_shared_probe_rows(kind):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1908_07628_gb300 import build
    build.build()
    import paper_1908_07628_gb300 as g
    n, f = 128, 1 if kind == "whole_scan" else 2
    wl = sp.random_workload(n=n, n_z=3, f=f, cell=6.4, n_sites=14, w=11, seed=41, scan_n=5,
                            n_types=2, alpha=0.02, beta=0.03, dz=1.8)
    if kind == "partly":       # a few positions of the sites repeated at other depths
        for a in (wl.site_x, wl.site_y):
            a[7:] = a[:7]
    want = lin.linear_map(wl)
    assert want.max() > 0
    ctx = g.Context(0)
    sm = g.build_smatrix_for(ctx, wl)
    for prec in ("tf32", "bf16x3"):
        for how in ("probe_first", "transition_first", "auto"):
            for cap in (0, 2):
                ctx.set_association(how)
                ctx.set_batch_sites(cap)
                got = g.inelastic_map_for(ctx, sm, wl, prec)
                assert np.linalg.norm(got - want) / np.linalg.norm(want) < EPS[prec], (prec, how, cap)
