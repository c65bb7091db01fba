"""The scan that solves the tridiagonal half of the implicit step (rd_scan.cuh),
modelled in float32 on the CPU and compared with a dense float64 solve: over
grid sizes, one or two segments per row, and ratios from no diffusion to a
decay length far beyond the domain."""
import numpy as np
import pytest

F = np.float32


def _coef(n, alpha, beta, mu):
    lam = F(beta * mu + alpha)
    if beta > 0:
        h = F(0.5) * (lam / beta)
        a = F(1) / (F(1) + (h + np.sqrt(h * h + (h + h))))
    else:
        a = F(0)
    om = F(1) - a
    sc = om * om / lam
    g = F(1) / (om * (F(1) + a))
    pw = [a]
    for _ in range(5):
        pw.append(pw[-1] * pw[-1])
    geo = F(1)
    for _ in range(1, n // 16):
        geo = geo * pw[5] + F(1)
    one_m = om
    for p in pw[:5]:
        one_m = one_m * (F(1) + p)
    return a, sc, g, F(a ** n), F(1) / (one_m * geo)


def _scan(n, ns, r, alpha, beta, mu):
    a, sc, g, an, inv = _coef(n, F(alpha), F(beta), F(mu))
    h = n // ns
    ah = F(a ** h)
    seg = [r[s * h:(s + 1) * h].astype(F) for s in range(ns)]
    lr = []
    for x in seg:
        L, R = x[-1], x[0]
        for m in range(1, h):
            L, R = a * L + x[h - 1 - m], a * R + x[m]
        lr.append((L, R))
    Lt, Rt = lr[-1][0], lr[0][1]
    if ns == 2:
        Lt, Rt = ah * Lt + lr[0][0], ah * Rt + lr[1][1]
    out = []
    for s, x in enumerate(seg):
        left, right = (an * Rt + Lt) * inv, (an * Lt + Rt) * inv
        if ns == 2 and s == 1:
            left = ah * left + lr[0][1]
        if ns == 2 and s == 0:
            right = ah * right + lr[1][0]
        f, acc = np.empty(h, F), left
        for m in range(h):
            acc = a * acc + x[m]
            f[m] = acc
        acc = (a * right + f[-1]) * g
        f[-1] = acc
        for m in range(h - 2, -1, -1):
            acc = a * acc + f[m]
            f[m] = acc
        out.append(f * sc)
    return np.concatenate(out)


@pytest.mark.parametrize("n", [16, 48, 64, 112, 128])
@pytest.mark.parametrize("beta", [0.0, 1e-3, 0.6, 41.0, 400.0, 1e5])
def test_scan_matches_dense_solve(n, beta):
    rng = np.random.default_rng(n)
    lap = np.diag(np.full(n, -2.0)) + np.diag(np.ones(n - 1), 1) + np.diag(np.ones(n - 1), -1)
    lap[0, 0] = lap[-1, -1] = -1.0
    beta = float(F(beta))
    for alpha in (1.0, float(F(1.0005))):
        for k in (0, 1, 3, n // 2, n - 1):
            mu = float(F(4 * np.sin(np.pi * k / (2 * n)) ** 2))
            r = (rng.standard_normal(n) + rng.standard_normal()).astype(F)
            lam = alpha + beta * mu
            want = np.linalg.solve(lam * np.eye(n) - beta * lap, r.astype(np.float64))
            for ns in (1, 2):
                got = _scan(n, ns, r, alpha, beta, mu)
                # the rounding of a acts like a relative change of beta of at most
                # 2^-23 / (1 - a), which moves x by no more than that share of it;
                # the recursions round once per node and decay over 1 / (1 - a) nodes
                a = float(_coef(n, F(alpha), F(beta), F(mu))[0])
                tol = 2.0**-23 * (4.0 + 2.0 * min(1.0 / (1.0 - a), n))
                err = np.linalg.norm(got - want) / np.linalg.norm(want)
                assert err <= tol, (n, ns, beta, k, err, tol)
