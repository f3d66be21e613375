"""Sums of lines with windows of their own: what is added at a point keeps its compensation however
the windows' ends alternate between the parts of a tile."""
import math

import numpy as np
import pytest

import synth
from oracle import kappa as okappa

pytestmark = pytest.mark.gpu
DNU = 1.0 / 64.0  # offsets in grid points are exact
T = 296.0         # the reference temperature: intensities are S_ref, widths gamma_ref
TILE = 2048       # first point of a tile


@pytest.fixture(scope="module")
def rt():
    import paper_cs_0703028_gb300 as m
    return m


def _lines(at, strength, gamma):
    """Lines at grid indices `at` (ascending) whose Lorentz wing is strength / (distance in points)^2."""
    n = len(at)
    u = 0.1 * 101325.0 / (1.380649e-23 * T) * 1e-6
    lines = synth.make_lines(n, 2000.0, 2001.0, synth.rng_for(51, 0))
    lines.nu0[:] = 2000.0 + np.asarray(at, dtype=float) * DNU
    lines.gamma_ref[:] = gamma
    lines.S_ref[:] = np.asarray(strength) * DNU * DNU * math.pi / (u * gamma)
    lines.E_lower[:] = 0.0
    lines.T_ref = T
    return lines


def _spec(kappa_min, cutoff=25.0):
    return synth.Spectral(nu_min=2000.0, dnu=DNU, n_nu=4096, cutoff=cutoff, profile="lorentz", nT=1, T_min=T, T_max=T, kappa_min=kappa_min)


# One strong line, its window cut at 1600 points, ends 120 points into a tile; 120 weak lines end
# there and 70 points into it by turns, each worth 0.45 to 0.47 units in the last place of the strong
# one: added to it one by one they vanish, all 60 together are 27 units.
# Tolerance on the weak lines' share: the strong line's value is the same bits in both tables, so what
# is left is the rounding of the two results (half a unit each) and of the weak sum: 2 units.
def test_window_ends_that_alternate_keep_their_sums(rt):
    B = 1.9  # the strong line's wing at its window's end
    unit = 2.0 ** -23
    weak = 0.45 * unit
    at = TILE - 1480 + np.concatenate([[0], np.arange(10, 130)])
    end = TILE + np.where(np.arange(121) % 2 == 0, 120, 70)
    w = end - at + 0.3
    lines = _lines(at, np.where(np.arange(121) == 0, B * 1600.0 ** 2, weak * w * w), 0.01)
    strong = lines.subset(np.array([0]))
    spec = _spec(weak)
    pts = slice(TILE + 96, TILE + 121)
    got = [rt.build_kappa(l, spec).cpu().numpy().astype(np.float64)[0, pts] for l in (strong, lines)]
    ref = [okappa.kappa_table(l, spec)[0, pts] for l in (strong, lines)]
    assert (ref[1] - ref[0] > 20 * unit).all() and (got[0] >= 1.0).all() and (got[0] < 2.0).all()
    assert np.max(np.abs((got[1] - got[0]) - (ref[1] - ref[0]))) <= 2 * unit


# A point's offset from a line centre is rounded once, so a lone line's value there is the same bits
# wherever the grid begins, whichever lane and place of it the point falls to.
@pytest.mark.parametrize("at,points", [(300.2718281828, 90.0), (700.4142135623, 25.0), (1023.4577215664, 120.0), (511.5772156649, 3.0)])
def test_lone_line_is_the_same_wherever_the_grid_begins(rt, at, points):
    lines = _lines([at], np.array([1e-2 * points ** 2]), 0.02)
    spec = _spec(1e-2, cutoff=4.0)
    ref = rt.build_kappa(lines, spec).cpu().numpy()[0]
    assert 2 * int(points) - 1 <= np.count_nonzero(ref) <= 2 * int(points) + 2
    for shift in (1, 2, 3, 5, 6, 7, 17, 100, 255):
        s = _spec(1e-2, cutoff=4.0)
        s.nu_min = 2000.0 + shift * DNU
        got = rt.build_kappa(lines, s).cpu().numpy()[0]
        assert np.array_equal(got[:spec.n_nu - shift], ref[shift:])
