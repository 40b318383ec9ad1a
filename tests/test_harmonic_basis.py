"""Expansions in the harmonic basis ((P + 1)^2 terms): every order and every chunking of the
right-hand sides against the float-float operator of the same tree, and the truncated sum itself
against the full Cartesian one on the CPU."""
import math

import numpy as np
import pytest

from paper_1812_10722_gb300 import inputs as I


def _index(a, b, c):
    n = a + b + c
    return n * n + (2 * n if c else n) - a


@pytest.mark.parametrize("P", [1, 2, 5, 8])
def test_basis_sums_the_cartesian_expansion(P):
    # sum over |k| <= P of a_k u^k (Cartesian, (P+1)(P+2)(P+3)/6 terms) = the harmonic terms' sum;
    # FP64 rounding of a few hundred terms bounded by |u|/|R| < 1: 1e-12
    rng = np.random.default_rng(P)
    terms = sorted(((_index(a, n - c - a, c), (a, n - c - a, c)) for n in range(P + 1) for c in (0, 1) if c <= n
                    for a in range(n - c + 1)))
    assert [t for t, _ in terms] == list(range((P + 1) ** 2))
    for _ in range(10):
        R, u = rng.normal(size=3), rng.normal(size=3)
        u *= 0.5 * np.linalg.norm(R) / np.linalg.norm(u)
        r2 = R @ R
        a = {(0, 0, 0): r2 ** -0.5}
        for n in range(1, P + 1):
            for i in range(n + 1):
                for j in range(n - i + 1):
                    k = (i, j, n - i - j)
                    lower = [tuple(np.subtract(k, np.eye(3, dtype=int)[d] * e)) for e in (1, 2) for d in range(3)]
                    s1 = sum(R[d] * a.get(lower[d], 0.0) for d in range(3))
                    s2 = sum(a.get(q, 0.0) for q in lower[3:])
                    a[k] = -((2 * n - 1) * s1 + (n - 1) * s2) / (n * r2)
        full = sum(v * np.prod(u ** np.array(k)) for k, v in a.items())
        g = np.zeros(len(terms))
        g[0] = 1.0
        for t, (i, j, c) in terms[1:]:
            p3 = g[_index(i, j, 0)] if c else -sum(g[_index(*q, 1)] for q in ((i - 2, j), (i, j - 2)) if min(q) >= 0)
            g[t] = (u[2] * p3 + (u[0] * g[_index(i - 1, j, c)] if i else 0.0)
                    + (u[1] * g[_index(i, j - 1, c)] if j else 0.0)) / (i + j + c)
        harm = sum(a[k] * math.factorial(k[0]) * math.factorial(k[1]) * g[t] for t, k in terms)
        assert abs(harm - full) < 1e-12 * abs(full)


@pytest.mark.gpu
@pytest.mark.parametrize("P,B", [(1, 1), (2, 8), (3, 9), (4, 17), (5, 16), (6, 33), (7, 1), (7, 8), (8, 32), (8, 35)])
def test_every_order_and_chunk(P, B):
    # FP32 against float-float: 1e-5, the bound of the FP32 operator; FP64 against float-float:
    # 1e-11, the float-float operator's bound
    from paper_1812_10722_gb300 import lspr
    v, t = I.icosphere(3, 10.0)
    keep = np.ones(len(t), bool)
    keep[::29] = False
    t = t[keep]
    x = I.random_complex(2 * len(t), seed=P, batch=B)
    s = I.drude_eps(np.linspace(360.0, 400.0, B)) / I.EPS_WATER
    with lspr.Context(0) as ctx:
        ctx.mesh_upload(v, t)
        ctx.tree_build(0.5, P, 40)
        assert ctx.info()["n_m2p_pairs"] > 0
        ref = ctx.matvec(x, s, "tree_ff")
        for mode, tol in (("tree_fp32", 1e-5), ("tree_fp64", 1e-11)):
            y = ctx.matvec(x, s, mode)
            for b in range(B):
                assert np.linalg.norm(y[b] - ref[b]) < tol * np.linalg.norm(ref[b]), (mode, b)
