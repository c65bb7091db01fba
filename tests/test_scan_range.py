"""Where the scan of the implicit solve ends (kScanMaxRatio of rd_scan.cuh) and the
elimination beyond it, modelled in float32 on the CPU and compared with a
float64 solve in the cosine basis: a dense float64 solve would itself lose about
2^-53 beta of the answer."""
import os
import re

import numpy as np
import pytest

from tests.test_scan_model import F, _scan

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1605_04718_gb300", "csrc")


def _max_ratio():
    with open(os.path.join(CSRC, "rd_scan.cuh")) as f:
        return float(re.search(r"kScanMaxRatio = ([0-9.e+]+)f?;", f.read()).group(1))


def _eliminate(n, r, alpha, beta, mu):
    """Pivots beta + e_i held as their excess e_i: sums of positive terms only."""
    alpha, beta, mu = F(alpha), F(beta), F(mu)
    lam = F(beta * mu + alpha)
    d, q = np.empty(n, F), np.empty(n, F)
    e, s, qp = F(0), F(0), F(0)
    for i in range(n):
        e = F(lam + e * qp)
        s = F(r[i] + qp * s)
        q[i] = qp = F(1) / (F(1) + e / beta)
        d[i] = s / (e if i == n - 1 else e + beta)
    for i in range(n - 2, -1, -1):
        d[i] = F(d[i] + q[i] * d[i + 1])
    return d


def _exact(n, r, alpha, beta, mu):
    k, i = np.arange(n)[:, None], np.arange(n)[None]
    c = np.cos(np.pi * k * (i + 0.5) / n) * np.sqrt(2 / n)
    c[0] = np.sqrt(1 / n)
    m = 4 * np.sin(np.pi * np.arange(n) / (2 * n)) ** 2
    alpha, beta, mu = (float(F(x)) for x in (alpha, beta, mu))
    return c.T @ ((c @ r.astype(np.float64)) / (alpha + beta * mu + beta * m))


def _rows(n, seed):
    rng = np.random.default_rng(seed)
    for k in (0, 1, 3, n // 2, n - 1):
        r = (rng.standard_normal(n) + 2.0 * rng.choice([-1.0, 1.0])).astype(F)
        yield float(F(4 * np.sin(np.pi * k / (2 * n)) ** 2)), r


# rounding: each sweep over n nodes adds at most n roundings of 2^-24 to its running
# sum (two sweeps, and the entering sums), relative to sums that do not cancel
def _tol(n):
    return 2.0**-24 * (4 * n + 16)


@pytest.mark.parametrize("n", [16, 32, 48, 64, 80, 128])
@pytest.mark.parametrize("alpha", [1.0, 0.5, 1.5])
def test_scan_holds_up_to_its_limit(n, alpha):
    for mu, r in _rows(n, n):
        beta = _max_ratio() * alpha
        want = _exact(n, r, alpha, beta, mu)
        for ns in (1, 2):
            got = _scan(n, ns, r, alpha, beta, mu)
            assert np.linalg.norm(got - want) <= _tol(n) * np.linalg.norm(want), (mu, ns)


def test_limit_keeps_one_minus_a_resolved():
    """1 - a is about sqrt(lam / beta): at the limit it must be many units of a's
    last place (2^-24), far from where a rounds to 1 and the row becomes NaN."""
    assert 1e6 <= _max_ratio() <= 2.0**34
    with np.errstate(all="ignore"):
        assert np.isnan(_scan(64, 2, np.ones(64, F), 1.0, 1e16, 0.0)).any()


@pytest.mark.parametrize("n", [16, 32, 48, 64, 80, 128])
@pytest.mark.parametrize("beta", [41.0, 1e5, 1e10, 1e12, 1e16, 1e25])
@pytest.mark.parametrize("alpha", [1.0, 0.01])
def test_elimination_holds_at_any_beta(n, beta, alpha):
    for mu, r in _rows(n, n + 1):
        want = _exact(n, r, alpha, beta, mu)
        got = _eliminate(n, r, alpha, beta, mu)
        assert np.linalg.norm(got - want) <= _tol(n) * np.linalg.norm(want), mu
