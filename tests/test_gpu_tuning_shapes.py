"""The autotuner's choices are kept per shape: maps of equal sizes whose sites share their
probe rows and maps whose sites do not are timed each for themselves."""
import dataclasses

import numpy as np
import pytest

import specimen as sp

pytestmark = pytest.mark.gpu


def test_shared_and_distinct_probe_rows_are_two_shapes():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1908_07628_gb300 import build
    build.build()
    import paper_1908_07628_gb300 as g
    # a scan of 16 x 16 positions over the whole cell: every window of cell / 2 holds 8 x 8
    n, cell, k = 128, 6.4, 8
    wl = sp.random_workload(n=n, n_z=2, f=2, cell=cell, n_sites=k, w=8, seed=5, alpha=0.02,
                            beta=0.03, dz=1.8)
    wl = wl.with_scan((16, 16, 0.0, 0.0, cell / 16, cell / 16))
    at = (np.arange(k) + 0.3) * cell / 16
    shared = dataclasses.replace(wl, site_x=np.full(k, at[0]), site_y=np.full(k, at[0]))
    distinct = dataclasses.replace(wl, site_x=at, site_y=at[::-1].copy())
    ctx = g.Context(0)
    sm = g.build_smatrix_for(ctx, wl)
    for maps, shapes in ((shared, 1), (distinct, 2), (shared, 2)):
        g.inelastic_map_for(ctx, sm, maps, "tf32")
        tuned = ctx.tuning_read()
        assert len(tuned) == shapes, tuned
        assert all(t["nr_max"] == 64 for t in tuned)
