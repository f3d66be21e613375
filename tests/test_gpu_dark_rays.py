"""Rays whose transmission has underflowed to zero only have their remaining visits counted.

The count in closed form is compared, ray by ray, with the walk itself: a call that records
its rays lists every cell, a call that does not counts.  Both must report the same number of
steps (integers, equal) and the same tallies up to the order of their binary64 sums (1e-12).
"""
import math

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    import paper_cs_0703028_gb300 as m
    return m


def _spec(n_nu=64, nT=5):
    return synth.Spectral(nu_min=2000.0, dnu=0.5, n_nu=n_nu, cutoff=25.0, profile="voigt", nT=nT, T_min=800.0, T_max=2000.0)


def _trace(rt, gs, spec, kap, ncells, n, record, **kw):
    t = rt.Tally(ncells)
    rec = rt.Record(n, record) if record else None
    rt.trace(gs, kap, spec, t, n, record=rec, **kw)
    ab, sc, _ = t.read()
    return ab, sc, int(t.steps[0]), rec


# axes of one cell, uneven boxes, a slab, odd cell sizes, the longest axis of the closed form
# and one longer (walked); the absorption makes rays dark within their first cells.  Two
# boxes of 2048 and 2049 cells, in a thin gas, have the largest tally kept in shared memory and
# the smallest that is not (a recorded trace's never is)
@pytest.mark.parametrize("dims,h,kappa", [
    ((1, 1, 1), (1.0, 1.0, 1.0), 200.0), ((1, 7, 300), (0.013, 0.013, 0.013), 400.0), ((33, 32, 31), (1 / 32,) * 3, 50.0),
    ((128, 3, 70), (0.01, 0.5, 0.02), 100.0), ((75, 52, 61), (1 / 75,) * 3, 30.0), ((64, 1, 1), (1 / 64, math.inf, math.inf), 100.0),
    ((5, 9, 1), (0.1, 0.1, math.inf), 100.0), ((16, 16, 8), (0.1, 0.1, 0.1), 0.05), ((683, 3, 1), (0.1, 0.1, 0.1), 0.05), ((3, 4, 5), (1e4, 1e4, 1e4), 1.0), ((65536, 1, 2), (1e-2, 1.0, 1.0), 500.0),
    ((65537, 1, 2), (1e-2, 1.0, 1.0), 500.0)])
def test_counted_visits_equal_walked_ones(rt, dims, h, kappa):
    import torch
    spec = _spec()
    nc = dims[0] * dims[1] * dims[2]
    rng = np.random.default_rng(3)
    g = synth.Grid(*dims, *h, rng.uniform(800.0, 2000.0, nc).astype(np.float32))
    gs, keep = rt.make_grid(g)
    kap = torch.from_numpy((kappa * rng.uniform(0.5, 2.0, (spec.nT, spec.n_nu))).astype(np.float32)).cuda()
    n = 400 if max(dims) > 1000 else 20000
    ab, sc, steps, _ = _trace(rt, gs, spec, kap, nc, n, 0, seed=5)
    abr, scr, stepsr, rec = _trace(rt, gs, spec, kap, nc, n, sum(dims) + 4, seed=5)
    assert steps == stepsr == int(rec.n_visits.sum())
    assert np.allclose(ab, abr, rtol=1e-12, atol=1e-12 * ab.max())
    assert np.allclose(sc[:3], scr[:3], rtol=1e-12)


def test_counted_visits_of_a_beam(rt):
    import torch
    spec = _spec()
    g = synth.uniform_grid(97, 3, 5, 0.02, 0.02, 0.02, 1000.0)
    gs, keep = rt.make_grid(g)
    kap = torch.full((spec.nT, spec.n_nu), 300.0, dtype=torch.float32, device="cuda")
    _, _, steps, _ = _trace(rt, gs, spec, kap, g.ncells, 64, 0, flags=rt.RT_SRC_BEAM)
    assert steps == 64 * 97


@pytest.mark.parametrize("walk", ["lbl", "mlp", "batch"])
def test_other_walks_count_the_same_visits(rt, walk):
    import torch
    spec = _spec(nT=4)
    g = synth.gaussian_hotspot_grid(13, 1.0, 800.0, 2000.0, 0.2, dims=(13, 8, 17))
    gs, keep = rt.make_grid(g)
    n = 3000
    kap = torch.full((spec.nT, spec.n_nu), 100.0, dtype=torch.float32, device="cuda")
    _, _, walked, _ = _trace(rt, gs, spec, kap, g.ncells, n, 60, seed=7)  # the rays' visits do not depend on kappa
    t = rt.Tally(g.ncells)
    if walk == "lbl":
        lines = synth.make_lines(400, 2000.0, 2032.0, np.random.default_rng(1))
        rt.trace_lbl(gs, lines, spec, t, n, seed=7)
    elif walk == "mlp":
        norm = rt.make_norm([math.log(2000.0), 800.0, 0.5, 0.01], [math.log(2032.0), 2000.0, 5.0, 0.3], 5.0, 0.5)
        rt.trace_mlp(gs, torch.from_numpy(synth.mlp_init(0, spread_biases=True)).cuda(), norm, spec, t, n, seed=7)
    else:
        b = rt.Batch([g], [n], spec, seed=7)
        b.trace(kap)
        t = b.tallies[0]
    t.read()
    assert int(t.steps[0]) == walked
