"""Best exponential sums for 1 / x: the generator of the tables in csrc/gr_quad.cuh (not needed to build or run the library).

`python -m paper_2511_15898_b200.quadrature K EPS` prints the sum of K terms

    1 / x = sum_k c_k exp(-t_k x)   on [1, R],   largest relative error EPS,

with the largest R for which there is one.  The error of the best sum equioscillates at 2 K + 1 points of the interval, both ends among them
(Braess and Hackbusch, Approximation of 1/x by exponential sums, 2005).  Remez exchange: Newton's method for equal errors of alternating
sign at given points, then the points move to the extrema.  At R = 1 the sum is the Gauss-Laguerre rule; from there R grows by factors in log R, the
start of each exchange extrapolated from the last two, until the error reaches EPS.  In mpmath, with digits enough for the cancellation.
"""
from __future__ import annotations

import sys

import numpy as np
from mpmath import cos, exp, log, lu_solve, matrix, mp, mpf, pi


def _laguerre(K):
    """Nodes and weights of the Gauss-Laguerre rule: Newton's method from the double precision nodes."""
    def values(n, x):
        a, b = mpf(1), 1 - x
        for k in range(1, n):
            a, b = b, ((2 * k + 1 - x) * b - k * a) / (k + 1)
        return b, a                                  # L_n, L_(n-1)
    nodes, weights = [], []
    for x in map(mpf, np.polynomial.laguerre.laggauss(K)[0]):
        step = mpf(1)
        while abs(step) > mpf(10) ** (8 - mp.dps):
            p, q = values(K, x)
            step = p * x / (K * (p - q))
            x -= step
        nodes.append(x)
        weights.append(x / ((K + 1) * values(K + 1, x)[0]) ** 2)
    return nodes, weights


def _equal_errors(lt, lc, E, points):
    """Newton's method for  x sum_k c_k exp(-t_k x) - 1 = +E, -E, ...  at the points, in log t, log c and E."""
    K = len(lt)
    for _ in range(30):
        A, b = matrix(2 * K + 1, 2 * K + 1), matrix(2 * K + 1, 1)
        for i, x in enumerate(points):
            sign, total = (-1) ** i, mpf(0)
            for k in range(K):
                term = x * exp(lc[k] - exp(lt[k]) * x)
                total += term
                A[i, k], A[i, K + k] = -x * exp(lt[k]) * term, term
            A[i, 2 * K], b[i] = -sign, 1 + sign * E - total
        d = lu_solve(A, b)
        size = max(abs(d[i]) for i in range(2 * K))
        damp = min(mpf(1), mpf("0.3") / size) if size > 0 else mpf(1)
        lt = [lt[k] + damp * d[k] for k in range(K)]
        lc = [lc[k] + damp * d[K + k] for k in range(K)]
        E += damp * d[2 * K]
        if size < mpf(10) ** (-mp.dps // 3):
            break
    return lt, lc, E


def _extrema(lt, lc, points):
    """Interior extrema of the error, one near every interior point (Newton's method in log x, held between its neighbours)."""
    out = [points[0]]
    for left, x, right in zip(points, points[1:], points[2:]):
        u, lim = log(x), (log(right) - log(left)) / 8
        for _ in range(40):
            x, f1, f2 = exp(u), mpf(0), mpf(0)
            for a, c in zip(lt, lc):
                tx = exp(a) * x
                term = x * exp(c - tx)
                f1 += (1 - tx) * term
                f2 += ((1 - tx) ** 2 - tx) * term
            step = max(-lim, min(lim, f1 / f2))
            u -= step
            if abs(step) < mpf(10) ** -12 * lim:
                break
        out.append(exp(u))
    out.append(points[-1])
    if any(b <= a for a, b in zip(out, out[1:])):
        raise ArithmeticError("extrema out of order")
    return out


def _remez(lt, lc, E, points):
    span = log(points[-1])
    for _ in range(25):
        lt, lc, E = _equal_errors(lt, lc, E, points)
        moved = _extrema(lt, lc, points)
        change = max(abs(log(b) - log(a)) for a, b in zip(points, moved))
        points = moved
        if change < mpf("1e-4") * span:
            break
    return log(points[-1]), lt, lc, E, points


def _between(a, b, s):
    """State at a + s (b - a) in log R: logarithms of nodes, coefficients and the error, relative places of the points."""
    lr = a[0] + s * (b[0] - a[0])
    mix = lambda x, y: [p + s * (q - p) for p, q in zip(x, y)]
    places = mix([log(x) / a[0] for x in a[4]], [log(x) / b[0] for x in b[4]])
    E = abs(a[3]) * exp(s * (log(abs(b[3])) - log(abs(a[3])))) * (1 if b[3] > 0 else -1)
    return mix(a[1], b[1]), mix(a[2], b[2]), E, [mpf(1)] + [exp(f * lr) for f in places[1:-1]] + [exp(lr)]


def best_sum(K, eps):
    """(R, t, c): the sum of K terms whose relative error on [1, R] is eps, t ascending."""
    mp.dps = 70 + 5 * K
    lr = {1: mpf("1e-5"), 2: mpf("1e-3"), 3: mpf("5e-3"), 4: mpf("0.01"), 5: mpf("0.02")}.get(K, mpf("0.05"))
    nodes, weights = _laguerre(K)
    start = ([log(x) - lr / 2 for x in nodes], [log(w) + x - lr / 2 for x, w in zip(nodes, weights)], mpf(0),
             [exp(lr * (1 - cos(pi * i / (2 * K))) / 2) for i in range(2 * K + 1)])
    last, here = None, _remez(*start)
    while abs(here[3]) < eps:
        grow, nxt = mpf("0.3"), None
        while nxt is None:
            try:
                if last is None:
                    f = 1 + grow
                    nxt = _remez(here[1], here[2], here[3], [exp(f * log(x)) for x in here[4]])
                else:
                    nxt = _remez(*_between(last, here, 1 + grow * here[0] / (here[0] - last[0])))
            except (ArithmeticError, ZeroDivisionError):
                grow /= 3
                if grow < mpf("1e-4"):
                    raise
        last, here = here, nxt
    # the error is between those of `last` and `here`
    while abs(abs(here[3]) / eps - 1) > mpf("1e-3"):
        s = (log(mpf(eps)) - log(abs(last[3]))) / (log(abs(here[3])) - log(abs(last[3])))
        mid = _remez(*_between(last, here, s))
        if abs(mid[3]) < eps and abs(abs(mid[3]) / eps - 1) > mpf("1e-3"):
            last = mid
        else:
            here = mid
    order = sorted(range(K), key=lambda k: here[1][k])
    return float(exp(here[0])), [float(exp(here[1][k])) for k in order], [float(exp(here[2][k])) for k in order]


if __name__ == "__main__":
    R, t, c = best_sum(int(sys.argv[1]), float(sys.argv[2]))
    print("R = %.7g" % R)
    for a, b in zip(t, c):
        print("{%.17g, %.17g}," % (a, b))
