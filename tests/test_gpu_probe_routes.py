"""Probe rows gathered once per distinct probe set and gathered per site with each batch, on
the same map: an operand budget too small for the sets turns the first into the second.

Tolerance: 1e-12, the order of the FP64 map sums (the operands are the same values)."""
import dataclasses

import numpy as np
import pytest

import specimen as sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["tf32", "bf16x3"])
@pytest.mark.parametrize("positions", [8, 12, 13])   # of 24 sites; 13 are not shared
def test_both_routes_give_one_map(prec, positions):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1908_07628_gb300 import build
    build.build()
    import paper_1908_07628_gb300 as g
    n, cell, k, scan = 256, 12.8, 24, 128
    wl = sp.random_workload(n=n, n_z=3, f=2, cell=cell, n_sites=k, w=11, seed=17, alpha=0.02,
                            beta=0.03, dz=1.8)
    # every window of cell / 2 holds 64 x 64 of 128 x 128 positions; eight sets of their probe
    # rows take more than a quarter of the smallest budget
    at = ((np.arange(k) % positions) + 0.3) * cell / scan
    wl = dataclasses.replace(wl.with_scan((scan, scan, 0.0, 0.0, cell / scan, cell / scan)),
                             site_x=at, site_y=at.copy())
    ctx = g.Context(0)
    ctx.set_tile_width(128)
    sm = g.build_smatrix_for(ctx, wl)
    for how in ("probe_first", "transition_first"):
        ctx.set_association(how)
        maps, shared = [], []
        for mib in (8192, 64):
            ctx.set_operand_budget(mib)
            ctx.profile_enable(True)
            maps.append(g.inelastic_map_for(ctx, sm, wl, prec))
            shared.append("tc_gather_sets" in ctx.profile_read())
            ctx.profile_enable(False)
        assert shared == [positions <= 12, False], (how, shared)
        assert maps[0].max() > 0
        assert np.linalg.norm(maps[0] - maps[1]) <= 1e-12 * np.linalg.norm(maps[1]), how
