"""Rounding of the operator outside the PML: its error against extended precision, measured
against the error of the plain order ((cc x_C + x_W) + x_E + x_S) + x_N with one FMA, on the
coefficients the kernel stores.

On superposed plane waves (what a residual b - A x is formed of) the result is a tenth of its
terms, so every rounding before the terms cancel counts: with two neighbour pairs, the centre
joined to one of them before they meet, three roundings of at most twice the wave's size stand
against the plain order's four, and the two errors are alike (1.1 allows for the binades they
fall in); with the four neighbours summed first, one rounding at four times that size makes it
1.35 to 1.5.  On white noise the pairs round less than the plain chain."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1508_02897_gb300.build import build  # noqa: E402

build()
from paper_1508_02897_gb300.solver import HelmholtzDDM  # noqa: E402

LD = np.longdouble


def _fma(a, b, c):
    """a b + c rounded once: the product as two doubles (Dekker), the sum in extended precision."""
    def split(x):
        t = x * 134217729.0
        h = t - (t - x)
        return h, x - h
    p = a * b
    (ah, al), (bh, bl) = split(a), split(b)
    e = ((ah * bh - p) + ah * bl + al * bh) + al * bl
    return ((LD(p) + LD(c)) + LD(e)).astype(np.float64)


def _waves(n, cells, rng):
    i, j = np.meshgrid(np.arange(n), np.arange(n))
    k = 2 * np.pi / cells
    x = np.zeros((n, n))
    for _ in range(24):
        t = rng.uniform(0, 2 * np.pi)
        x += rng.normal() * np.cos(k * (np.cos(t) * i + np.sin(t) * j) + rng.uniform(0, 2 * np.pi))
    return x


@pytest.mark.parametrize("N,npml,medium", [(333, 8, "homogeneous"), (300, 4, "random")])
def test_operator_rounding(N, npml, medium):
    n, h = N + 2 * npml, 1.0 / N
    c = np.ones((n, n)) if medium == "homogeneous" else W.velocity_random_field(N, npml, seed=3)
    rng = np.random.default_rng(5)
    for cells, bound in ((10, 1.1), (14, 1.1), (20, 1.1), (0, 1.0)):
        om = 2 * np.pi * float(c.min()) * N / (cells or 10)
        s = HelmholtzDDM(N, npml, om, c, 2, 2, 0, factor=False)
        x = _waves(n, cells, rng) if cells else rng.normal(size=(n, n))
        y = s.matvec(torch.from_numpy(x.astype(np.complex128))).cpu().numpy().real
        s.close()
        k = om / c
        cc = (h * h) * (k * k) + -4.0
        o = slice(npml, n - npml)
        t = lambda dj, di: x[npml + dj:n - npml + dj, npml + di:n - npml + di]
        xc, xw, xe, xs, xn, cc = t(0, 0), t(0, -1), t(0, 1), t(-1, 0), t(1, 0), cc[o, o]
        exact = LD(cc) * LD(xc) + ((LD(xw) + LD(xe)) + (LD(xs) + LD(xn)))
        plain = ((_fma(cc, xc, xw) + xe) + xs) + xn
        err = float(np.sqrt(np.sum((y[o, o] - exact) ** 2)))
        ref = float(np.sqrt(np.sum((plain - exact) ** 2)))
        assert err <= bound * ref, (cells, err / ref)
