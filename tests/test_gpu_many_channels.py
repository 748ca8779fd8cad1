"""FP32 maps of more channels than one launch takes.  With windows of one pixel and H a power
of two every product and sum of a channel is that of H = 1 scaled by it, so its map is |H|^2
times that of H = 1 bit for bit (one site, two groups of detector beams: the FP64 sum of two
values does not depend on their order)."""
import numpy as np
import pytest

import specimen as sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("types", [32767, 33000])   # 65534 and 66000 groups of 64 beams
def test_channels_past_one_launch(types):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1908_07628_gb300 import build
    build.build()
    import paper_1908_07628_gb300 as g
    n, cell, lam = 64, 6.4, sp.LAM_200KEV
    wl = sp.random_workload(n=n, n_z=2, f=1, cell=cell, n_sites=1, w=1, seed=8, scan_n=2,
                            alpha=lam * 1.2 / cell, beta=lam * 5.1 / cell, dz=1.8, n_types=1)
    assert 64 < g.count_beams(n, cell, lam, 1, wl.beta) <= 128
    rng = np.random.default_rng(9)
    h = (rng.choice([-1, 1], types) * 2.0 ** rng.integers(-4, 5, types)).astype(np.complex64)
    ctx = g.Context(0)
    sm = g.build_smatrix_for(ctx, wl)
    one = g.inelastic_map_for(ctx, sm, wl, "fp32", H=np.ones((1, 1, 1), np.complex64))
    got = g.inelastic_map_for(ctx, sm, wl, "fp32", H=h.reshape(types, 1, 1))
    want = (np.abs(h.astype(np.complex128)) ** 2)[:, None, None] * one
    assert want.min() > 0
    assert np.array_equal(got, want)
