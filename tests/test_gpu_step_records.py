"""The table walk steps on 8-byte cell records (position in the node grid, density scale), the
batched walk on whole ones: the same rays, so the same tallies up to the order of their binary64
sums (1e-12), for temperatures inside, on and beyond the table's nodes.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


# no, one, two and many brackets; node-pair and (n_nu nT above 64 MiB of pairs) wavenumber-major
# tables; a tally of few cells and one of many
@pytest.mark.parametrize("nT,n_nu,side,px", [(1, 50, 14, True), (2, 50, 14, False), (3, 64, 9, True), (33, 1000, 14, True),
                                             (90, 100000, 14, False), (64, 333, 20, True)])
def test_step_records_equal_whole_ones(nT, n_nu, side, px):
    import torch
    import paper_cs_0703028_gb300 as rt
    spec = synth.Spectral(nu_min=2000.0, dnu=0.01, n_nu=n_nu, cutoff=25.0, profile="voigt", nT=nT, T_min=800.0,
                          T_max=800.0 if nT == 1 else 2000.0)
    rng = np.random.default_rng(nT)
    nc = side * (side + 1) * (side - 1)
    T = rng.uniform(500.0, 2500.0, nc).astype(np.float32)
    T[::5] = rng.choice(np.linspace(800.0, 2000.0, max(nT, 2)), T[::5].size).astype(np.float32)
    g = synth.Grid(side, side + 1, side - 1, 0.1, 0.1, 0.1, T)
    if px:
        g.p_atm = rng.uniform(0.5, 2.0, nc).astype(np.float32)
        g.x = rng.uniform(0.05, 0.3, nc).astype(np.float32)
    kap = torch.from_numpy(rng.uniform(0.005, 0.05, (nT, n_nu)).astype(np.float32)).cuda()
    gs, keep = rt.make_grid(g)
    t = rt.Tally(nc)
    rt.trace(gs, kap, spec, t, 30000, seed=9)
    b = rt.Batch([g], [30000], spec, seed=9)
    b.zero()
    b.trace(kap)
    ab, sc, _ = t.read()
    abb, scb, _ = b.tallies[0].read()
    assert int(t.steps[0]) == int(b.tallies[0].steps[0])
    assert np.allclose(ab, abb, rtol=1e-12, atol=1e-12 * ab.max())
    assert np.allclose(sc[:3], scb[:3], rtol=1e-12)
