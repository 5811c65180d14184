"""Moment sums and normal equations of a regression in exact rational
arithmetic, from the double-precision features of the paths, and the error a
double-precision fit of them may have."""
from fractions import Fraction

import numpy as np

EPS = 2.0**-53
_SHIFT = 140  # doubles above 2^-87 as whole multiples of 2^-140
# (powers of x, w, y) in the order of the sums, and the basis functions
UNITS = {"s2": [(1, 0, 0), (2, 0, 0), (3, 0, 0), (4, 0, 0), (0, 0, 1), (1, 0, 1), (2, 0, 1)],
         "sv2": [(1, 0, 0), (2, 0, 0), (3, 0, 0), (4, 0, 0), (0, 1, 0), (1, 1, 0), (2, 1, 0),
                 (3, 1, 0), (0, 2, 0), (1, 2, 0), (2, 2, 0), (0, 3, 0), (1, 3, 0), (0, 4, 0),
                 (0, 0, 1), (1, 0, 1), (2, 0, 1), (0, 1, 1), (1, 1, 1), (0, 2, 1)]}
BASIS = {"s2": [(0, 0), (1, 0), (2, 0)],
         "sv2": [(0, 0), (1, 0), (2, 0), (0, 1), (1, 1), (0, 2)]}


def whole(a):
    """doubles as Python integers in units of 2^-_SHIFT"""
    out = []
    for v in np.asarray(a, dtype=float):
        n, d = float(v).as_integer_ratio()
        q, r = divmod(n << _SHIFT, d)
        assert r == 0, v
        out.append(q)
    return np.array(out, dtype=object)


def feature(v, scale):
    """fma(v, scale, -1) in double, from the exact value"""
    c = Fraction(float(scale))
    return np.array([float(Fraction(float(t)) * c - 1) for t in v])


def moments(x, w, y, basis):
    """{(a, b, c): exact sum of x^a w^b y^c}"""
    X, W, Y = whole(x), whole(w), whole(y)
    out = {(0, 0, 0): Fraction(len(x))}
    px, pw = [1, X, X * X, X * X * X, X * X * X * X], [1, W, W * W, W * W * W, W * W * W * W]
    for a, b, c in UNITS[basis]:
        s = px[a] * pw[b] * (Y if c else 1)
        out[a, b, c] = Fraction(int(s.sum()), 1 << (_SHIFT * (a + b + c)))
    return out


def solve(m, basis):
    """exact coefficients of the normal equations with the moments m"""
    f = BASIS[basis]
    n = len(f)
    A = [[m[p[0] + q[0], p[1] + q[1], 0] for q in f] + [m[p[0], p[1], 1]] for p in f]
    for k in range(n):
        for i in range(k + 1, n):
            t = A[i][k] / A[k][k]
            A[i] = [a - t * b for a, b in zip(A[i], A[k])]
    beta = [Fraction(0)] * n
    for i in reversed(range(n)):
        beta[i] = (A[i][n] - sum(A[i][j] * beta[j] for j in range(i + 1, n))) / A[i][i]
    return beta


def smallest_pivot(m, basis):
    """the smallest pivot of the Gram matrix over its largest diagonal entry:
    at 1e-13 or below the library takes the regression for singular"""
    f = BASIS[basis]
    A = [[m[p[0] + q[0], p[1] + q[1], 0] for q in f] for p in f]
    top = max(A[i][i] for i in range(len(f)))
    low = top
    for k in range(len(f)):
        low = min(low, A[k][k])
        for i in range(k + 1, len(f)):
            t = A[i][k] / A[k][k]
            A[i] = [a - t * b for a, b in zip(A[i], A[k])]
    return float(low / top)


def scaled_error(beta, ref, m, basis):
    """|D (beta - ref)|, D the square roots of the Gram matrix' diagonal"""
    d = [float(m[2 * p[0], 2 * p[1], 0]) ** 0.5 for p in BASIS[basis]]
    return float(np.linalg.norm([s * float(Fraction(float(b)) - r)
                                 for s, b, r in zip(d, beta, ref)]))


def error_bound(m, y, ref, basis):
    """What scaled_error of a double-precision fit may be: the condition number
    of the Gram matrix scaled to unit diagonal (Cholesky's error, and the
    effect of relative errors of the sums, grow with it) times 100 roundings of
    |D beta| + |y| (B (B + 1) = 42 of a Cholesky solve with 6 functions, the
    rest for the sums)."""
    f = BASIS[basis]
    d = np.array([float(m[2 * p[0], 2 * p[1], 0]) ** 0.5 for p in f])
    G = np.array([[float(m[p[0] + q[0], p[1] + q[1], 0]) for q in f] for p in f])
    cond = np.linalg.cond(G / d[:, None] / d[None, :])
    size = np.linalg.norm([s * float(b) for s, b in zip(d, ref)]) + np.linalg.norm(y)
    return 100.0 * EPS * cond * size, cond
