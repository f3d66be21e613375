"""bench.py's count of the values the line sum evaluates (no device involved)."""
import importlib.util
import os
import re

import numpy as np
import pytest

import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_line_sum", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_constants_are_the_kernels(bench):
    src = open(os.path.join(ROOT, "paper_cs_0703028_gb300", "csrc", "rt_kappa.cu")).read()
    want = tuple(int(re.search(r"\b%s = (\d+)[,;]" % k, src).group(1)) for k in ("kDist8", "kDist16", "kDistEdge"))
    here = open(os.path.join(ROOT, "bench.py")).read()
    assert tuple(int(v) for v in re.search(r"dist8, dist16, edge = 256, (\d+), (\d+), (\d+)", here).groups()) == want


# one line: every point of the tile it lies in, 16 nodes of the next tiles, 8 of the ones further out
def test_a_lone_line(bench):
    lines = synth.make_lines(1, 2000.0, 2001.0, synth.rng_for(61, 0))
    spec = synth.Spectral(nu_min=2000.0, dnu=0.01, n_nu=2560, cutoff=50.0, profile="lorentz", nT=3, T_min=500.0, T_max=900.0)
    lines.nu0[:] = 2000.0 + 0.01 * 1400.3  # tile 5 of 10, 120 points from tile 4 and 136 from tile 6
    far, core = bench.line_sum_values(lines, spec)
    assert core == {}
    # tiles 0, 1 and 9 are at least 704 points away, 2, 3, 7 and 8 at least 141, 4 to 6 nearer
    assert far == 3 * (8 * 3 + 16 * 4 + 256 * 3)


def test_no_more_values_than_pairs(bench):
    from oracle import kappa as okappa
    lines = synth.make_lines(400, 2000.0, 2100.0, synth.rng_for(61, 1))
    spec = synth.Spectral(nu_min=2000.0, dnu=0.01, n_nu=10000, cutoff=25.0, profile="voigt", nT=2, T_min=500.0, T_max=900.0)
    far, core = bench.line_sum_values(lines, spec)
    assert 0 < far < 0.2 * okappa.profile_evals(lines, spec)
    r = bench.line_sum_roofline([lines], spec, 1.0, {"fma_lane_ops_per_s": 1e13, "rcp_lane_ops_per_s": 1e12})
    assert r["frac"] == pytest.approx(max((6 * far + sum(v * (18 + 4 * (t - 1)) for t, v in core.items())) / 1e10,
                                          (far + sum(core.values())) / 1e9))
    assert np.isfinite(r["other_pipe_frac"])
