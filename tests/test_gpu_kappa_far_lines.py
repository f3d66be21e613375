"""The line sum's interpolated far lines against the binary64 oracle.

Far lines are summed at Chebyshev nodes of each 256-point tile (or 32-point sub-block, where
a window ends in the tile) and interpolated; these cases put window ends, grid tails and
empty ranges at the places where the split of the lines changes.

Tolerance: a value's binary32 roundings (at most ten in the prefactor, 6e-7; 2.2e-6 for the
rational series near a centre; two of a sum), plus 5e-8 for the interpolation: below 5e-6.
"""
import numpy as np
import pytest

import synth
from oracle import kappa as okappa

pytestmark = pytest.mark.gpu
TOL = 5e-6


@pytest.fixture(scope="module")
def rt():
    import paper_cs_0703028_gb300 as m
    return m


def _check(rt, lines, spec):
    got = rt.build_kappa(lines, spec).cpu().numpy().astype(np.float64)
    ref = okappa.kappa_table(lines, spec)
    nz = ref > 0
    assert np.array_equal(got > 0, nz)
    assert nz.any()
    assert (np.abs(got[nz] - ref[nz]) / ref[nz]).max() <= TOL


# one point, one tile less and more a point, a tail of a few points, of a whole sub-block, and
# tiles that every kind of line reaches
@pytest.mark.parametrize("n_nu", [1, 255, 256, 257, 290, 2048 + 32, 4099])
@pytest.mark.parametrize("profile,dnu,cutoff,nT", [("voigt", 0.02, 25.0, 2), ("voigt", 0.006, 25.0, 1), ("lorentz", 0.02, 25.0, 1),
                                                   ("voigt", 0.01, 4.0, 9), ("lorentz", 0.01, 9.6, 2)])
def test_far_lines_match_oracle(rt, n_nu, profile, dnu, cutoff, nT):
    span = n_nu * dnu
    rng = synth.rng_for(31, n_nu)
    lines = synth.make_lines(260, 2000.0 - 1.2 * cutoff, 2000.0 + span + 1.2 * cutoff, rng)
    spec = synth.Spectral(nu_min=2000.0, dnu=dnu, n_nu=n_nu, cutoff=cutoff, profile=profile, nT=nT, T_min=500.0,
                          T_max=500.0 if nT == 1 else 1100.0)
    _check(rt, lines, spec)


# window ends on the first and last point of tiles and sub-blocks, to one side of the tile
@pytest.mark.parametrize("side", [-1, 1])
def test_window_ends_at_every_place_of_a_tile(rt, side):
    dnu, cutoff = 0.015625, 25.0  # 1600 points: the offsets below are exact in binary64
    ends = np.array([0, 1, 31, 32, 33, 63, 64, 127, 128, 223, 224, 254, 255, 256, 257])
    base = 2000.0 + 512 * dnu if side < 0 else 2000.0 + 256 * dnu
    lines = synth.make_lines(ends.size, 2000.0, 2001.0, synth.rng_for(32, 0))
    lines.nu0[:] = np.sort(base + ends * dnu + side * cutoff)
    spec = synth.Spectral(nu_min=2000.0, dnu=dnu, n_nu=1024, cutoff=cutoff, profile="lorentz", nT=1, T_min=700.0, T_max=700.0)
    _check(rt, lines, spec)


# more lines than one staged chunk of any kind, and lines at one place
def test_many_lines_per_tile(rt):
    lines = synth.make_lines(3000, 1990.0, 2012.0, synth.rng_for(33, 0))
    lines.nu0[1000:1400] = lines.nu0[1000]
    spec = synth.Spectral(nu_min=2000.0, dnu=0.004, n_nu=520, cutoff=9.0, profile="voigt", nT=1, T_min=600.0, T_max=600.0)
    _check(rt, lines, spec)


# Windows per line and node: odd and even line counts and nodes (the windows' copies are
# aligned to pairs), thresholds from keeping everything to next to nothing, intensities and
# partition exponents that leave the binary32 estimate's range.  The evaluation counts are
# integers and equal.
@pytest.mark.parametrize("n,nT,kappa_min,profile,S,q_exp", [
    (301, 1, 1e-2, "voigt", 1e-20, 1.0), (300, 9, 1.0, "voigt", 1e-20, 1.0), (77, 3, 1e-6, "lorentz", 1e-20, 1.0),
    (301, 8, 30.0, "lorentz", 1e-19, 1.0), (128, 2, 1e-24, "voigt", 1e-40, 1.0), (65, 2, 1e-3, "voigt", 1e-20, 30.0),
    (1, 1, 1e-1, "voigt", 1e-20, 1.0)])
def test_adaptive_windows_match_oracle(rt, n, nT, kappa_min, profile, S, q_exp):
    import torch
    rng = synth.rng_for(34, n)
    lines = synth.make_lines(n, 1995.0, 2035.0, rng, S_lo=S, S_hi=30.0 * S)
    lines.q_exp = q_exp
    spec = synth.Spectral(nu_min=2000.0, dnu=0.01, n_nu=3001, cutoff=20.0, profile=profile, nT=nT, T_min=400.0,
                          T_max=400.0 if nT == 1 else 900.0, kappa_min=kappa_min)
    ev = torch.zeros(1, dtype=torch.int64, device="cuda")
    got = rt.build_kappa(lines, spec, evals=ev).cpu().numpy().astype(np.float64)
    ref = okappa.kappa_table(lines, spec)
    assert int(ev) == okappa.profile_evals(lines, spec)
    if S < 1e-38:
        return  # the values themselves are below binary32's range there
    assert np.array_equal(got > 0, ref > 0)
    nz = ref > 0
    assert nz.any()
    # an exponent of 30 multiplies the rounding of T_ref / T, 1.2e-7, into the ratio
    assert (np.abs(got[nz] - ref[nz]) / ref[nz]).max() <= (TOL if q_exp == 1.0 else 4.0 * TOL)
