"""The series that later iterations' lambda passes rest on (Sec. 3.2, Eq. 11),
checked on the CPU in FP64.

With t = c / (a + c), x = 2 t - 1 and e = tanh(ln(lambda / c) / 2),
sum_b r lambda^2 / (a + lambda)^2 = (1 + e)^2 sum_k (k + 1) (-e)^k N_k with
N_k = sum_b r t^2 x^k <= N_0, so the terms from k = K on add up to at most
(K + 1) |e|^K N_0 (1 + e)^2 / (1 - |e|)^2 whatever the spectrum: that bound
decides on the GPU whether a root is accepted.  These tests restate the series (not the GPU
code)."""
import numpy as np
import pytest

K = 8  # moments per pass


def spectra(kind, rng, n=4000):
    if kind == "wide":
        a = 10.0 ** rng.uniform(-12, 0, n)
    elif kind == "zeros":
        a = np.concatenate([np.zeros(n // 10), 10.0 ** rng.uniform(-8, 0, n)])
    else:
        a = 10.0 ** rng.uniform(-3, -2, n)
    return a, rng.exponential(1.0, a.size)


def f(lam, a, r):
    return np.sum(r * (lam / (a + lam)) ** 2)


def series(e, a, r, c):
    t = c / (a + c)
    x = 2.0 * t - 1.0
    return (1 + e) ** 2 * sum((k + 1) * (-e) ** k * np.sum(r * t * t * x ** k) for k in range(K))


@pytest.mark.parametrize("kind", ["wide", "zeros", "narrow"])
@pytest.mark.parametrize("s", [1e-3, 0.02, 0.1, 0.22, 0.7, -0.02, -0.22, -0.7])
def test_truncation_bound(kind, s):
    rng = np.random.default_rng(1)
    for c in 10.0 ** rng.uniform(-8, 0, 8):
        a, r = spectra(kind, rng)
        e = np.tanh(s / 2)
        n0 = np.sum(r * (c / (a + c)) ** 2)
        exact = f(c * np.exp(s), a, r)
        bound = (K + 1) * abs(e) ** K * n0 * (1 + e) ** 2 / (1 - abs(e)) ** 2
        assert abs(series(e, a, r, c) - exact) <= bound + 1e-13 * exact


@pytest.mark.parametrize("kind", ["wide", "zeros", "narrow"])
def test_root_near_the_centre(kind):
    """Within 2 % of the centre (iterations 5 on of the batched workload) the
    series' root is the root of Eq. 11 to 1e-12."""
    rng = np.random.default_rng(2)
    for c in 10.0 ** rng.uniform(-6, -1, 8):
        a, r = spectra(kind, rng)
        lam = c * np.exp(rng.uniform(-0.02, 0.02))
        T = f(lam, a, r)
        lo, hi = -0.05, 0.05
        for _ in range(80):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if series(mid, a, r, c) < T else (lo, mid)
        e = 0.5 * (lo + hi)
        assert abs(c * (1 + e) / (1 - e) / lam - 1) < 1e-12
