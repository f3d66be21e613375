"""The line sum's two approximations, evaluated in binary64 from the constants of its source: the
interpolation of far lines from the nodes of a tile, at the nearest distance each kind admits, and
Weideman's series with fewer terms, from the y on where each number of terms is used.  Neither may
change a line's value by more than half of one binary32 rounding, 2^-25."""
import os
import re

import numpy as np
import pytest

BOUND = 2.0 ** -25
SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_cs_0703028_gb300", "csrc",
                        "rt_kappa.cu")).read()


def _const(name):
    return float(re.search(r"\b%s = ([0-9.]+)f?[,;]" % name, SRC).group(1))


def _nodes(m):
    body = re.search(r"kNodes%d\{\{([^}]*)\}\}" % m, SRC).group(1)
    v = np.array([float(t) for t in body.split(",")])
    assert v.size == m
    return v


def _weights(nodes, at):
    w = np.ones((at.size, nodes.size))
    for m in range(nodes.size):
        for q in range(nodes.size):
            if q != m:
                w[:, m] *= (at - nodes[q]) / (nodes[m] - nodes[q])
    return w


# a centre is up to half a grid step nearer than its nearest grid point
@pytest.mark.parametrize("kind,points", [("kDist8", 256), ("kDist16", 256), ("kDistEdge", 32)])
@pytest.mark.parametrize("g", [0.0, 1.0, 5.0, 20.0, 100.0, 1000.0])
def test_interpolated_lines(kind, points, g):
    at = np.arange(float(points))
    if kind == "kDistEdge":
        nodes = _nodes(4)
        w = _weights(nodes, at)
    else:
        nodes = _nodes(16)
        w = _weights(nodes, at)
        if kind == "kDist8":  # 8 nodes' values are carried to the 16 nodes first
            w = w @ _weights(_nodes(8), nodes)
            nodes = _nodes(8)
    d = _const(kind) - 0.5
    worst = 0.0
    for centre in (-d, points - 1 + d, -1.5 * d, -4.0 * d):
        value = lambda u: 1.0 / ((u - centre) ** 2 + g * g)  # noqa: E731
        worst = max(worst, np.max(np.abs(w @ value(nodes) / value(at) - 1.0)))
    assert worst <= BOUND


def _series(n):
    """Weideman's (1994) L and coefficients of n terms, by the trapezoidal Fourier sums."""
    L, m = np.sqrt(n / np.sqrt(2.0)), 2 * n
    th = np.arange(-m + 1, m) * np.pi / m
    t = L * np.tan(th / 2.0)
    psi = np.exp(-t * t) * (L * L + t * t)
    return L, np.array([(psi * np.cos(k * th)).sum() / (2 * m) for k in range(1, n + 1)])


@pytest.mark.parametrize("n,name", [(16, "kTerms16"), (12, "kTerms12")])
def test_fewer_terms_of_the_rational_series(n, name):
    from scipy.special import wofz
    L, a = _series(n)
    for y in np.linspace(_const(name), 8.0, 60)[:-1]:
        z = np.linspace(0.0, np.sqrt(64.0 - y * y), 2001) + 1j * y
        Z = (L + 1j * z) / (L - 1j * z)
        w = 2.0 * np.polyval(a[::-1], Z) / (L - 1j * z) ** 2 + 1.0 / np.sqrt(np.pi) / (L - 1j * z)
        assert np.max(np.abs(w.real / wofz(z).real - 1.0)) <= BOUND, y
