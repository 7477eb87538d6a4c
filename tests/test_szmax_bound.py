"""The float bound on SZ that a queued close works with is never below the
largest SZ that Eq. 4 reports in double, so no hit is missed: the same float
arithmetic with each logarithm and exponential one unit in the last place off
either way, over the parameter space."""
import numpy as np
import pytest


def _szmax(g, r, k, theta, zr):
    """the largest sz with -g ln(sz / (g - g psi^r)) >= theta, -1 for none"""
    G = float(g) * 2.0 ** k
    psi = -np.expm1(np.log(zr.astype(np.float64) / G).mean())
    top = g - g * psi ** r
    sz = np.arange(g + 1, dtype=np.float64)
    with np.errstate(divide="ignore", invalid="ignore"):
        ok = -float(g) * np.log(sz / top) >= theta
    return int(np.flatnonzero(ok).max()) if ok.any() else -1


def _bound(g, r, k, theta, zr, ulp):
    f = np.float32
    off = lambda x: np.nextafter(x, f(np.inf) * f(ulp)) if ulp else x
    x = zr.astype(f) / (f(g) * f(2.0 ** k))
    ln = [off(np.log(v)) for v in x] + [f(0)] * (8 - r)
    for o in (4, 2, 1):  # the order of the kernel's sum over eight lanes
        ln = [f(ln[i] + ln[i ^ o]) for i in range(8)]
    psi = f(-off(np.expm1(f(ln[0] / f(r)))))
    pr = psi
    for _ in range(1, r):
        pr = f(pr * psi)
    xfac = f(np.exp(-theta / g))
    return int(max(f(0), f(f(f(f(g) - f(f(g) * pr)) * xfac) + f(0.01))))


@pytest.mark.parametrize("seed", range(6))
def test_bound_covers_the_reported_sizes(seed):
    rng = np.random.default_rng(seed)
    above = 0
    for _ in range(700):
        g = 1 << int(rng.integers(5, 13))
        r = int(rng.integers(3, 9))
        k = int(rng.integers(5, 25))
        theta = float(g * np.exp(rng.uniform(-9, 2.2)))
        full = (1 << k) * g
        # rows from empty to nearly saturated
        share = np.exp(-np.exp(rng.uniform(-12, 3)))
        zr = np.maximum(1, (full * share * rng.uniform(0.9, 1.0, r)).astype(np.uint64))
        sz = _szmax(g, r, k, theta, zr)
        for ulp in (-1, 0, 1):
            b = _bound(g, r, k, theta, zr, ulp)
            assert b >= sz, (g, r, k, theta, zr, ulp)
            above = max(above, b - max(sz, 0))
    assert above <= 1
