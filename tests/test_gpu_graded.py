"""Accuracy of the binary64 products on rows graded over many powers of two.

The tensor cores' products carry an error relative to the largest entries of the
two rows multiplied, K 2^-60 max|a| max|b|; FMAs (chol_options.fp64_products)
one relative to the sum's own terms, K 2^-53 sum |a_k b_k|, which is far smaller
where the large entries of one row meet the small ones of the other. Both bounds
are stated here on entries of L that are nothing but one such product.
"""
from fractions import Fraction

import numpy as np
import pytest

import gridgen
import oracle
from gpu_util import run
from lib_fixture import chol

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _opts(fp64, mode=0):
    o = chol().chol_default_options()
    o.small_max_cols = o.small_max_panel = 1
    o.fp64_products, o.update_mode = fp64, mode
    return o


def _graded(K, m, span, seed):
    """G (m x K): row 0 falls from 1 to 2^-span along the columns, the others rise."""
    rs = np.random.RandomState(seed)
    w = np.ldexp(1.0, -np.round(span * np.arange(K) / (K - 1)).astype(int))
    G = rs.uniform(0.5, 1.0, (m, K)) * w[::-1]
    G[0] = rs.uniform(0.5, 1.0, K) * w
    return G


def _problem(kind, G):
    """L has G below an identity, and right of it a column that starts with row 0's
    pivot: its entries are -(G G^T)_i0 / L_00. kind "trailing": one dense supernode
    (trailing update of a 64-column block); "update": G is the off-diagonal block of
    a leaf (U_J), beside a second leaf so that the separator is a supernode of its own."""
    m, K = G.shape
    n = K + m if kind == "trailing" else K + 2 + m
    A, pat = np.zeros((n, n)), np.ones((n, n), bool)
    r0 = n - m
    A[np.arange(r0), np.arange(r0)] = 1.0
    A[r0:, :K] = G
    A[np.arange(r0, n), np.arange(r0, n)] = 4.0 * np.abs(G @ G.T).sum(axis=1)
    if kind == "update":
        pat[K:K + 2, :K] = False
    cols, rows = np.nonzero((np.tril(np.ones((n, n), bool)) & pat).T)
    cp = np.concatenate([[0], np.cumsum(np.bincount(cols, minlength=n))]).astype(np.int64)
    return dict(n=n, colptr=cp, rowind=rows.astype(np.int32), values=A[rows, cols],
                perm=np.arange(n, dtype=np.int32)), r0


@pytest.mark.parametrize("kind,K", [("trailing", 64), ("update", 70), ("update", 200)])
@pytest.mark.parametrize("span", [0, 20, 60])
@pytest.mark.parametrize("mode", [0, 1])
def test_fill_entries(kind, K, span, mode):
    m = 100
    G = _graded(K, m, span, 3 * K + span)
    p, r0 = _problem(kind, G)
    far = np.arange(64, m)               # rows past the next diagonal block (which FMAs update)
    exact = [sum(Fraction(x) * Fraction(y) for x, y in zip(G[i], G[0])) for i in far]
    prod = np.array([float(e) for e in exact])
    terms = np.abs(G[far]) @ np.abs(G[0])
    top = np.abs(G[far]).max(axis=1) * np.abs(G[0]).max()
    for fp64, bound in ((0, K * 2.0 ** -60 * top), (1, K * U * terms)):
        got = run(p, None, _opts(fp64, mode))
        assert got["rc"] == 0
        lp, li, lx = got["L"]
        col = np.zeros(p["n"])
        col[li[lp[r0]:lp[r0 + 1]]] = lx[lp[r0]:lp[r0 + 1]]
        s00 = float(Fraction(p["values"][p["colptr"][r0]]) - sum(Fraction(x) ** 2 for x in G[0]))
        # the root, its reciprocal and the products with it: 8 u; S_00 itself K u
        err = np.abs(col[r0 + far] * np.sqrt(s00) + prod)
        assert np.all(err <= bound + (K + 8) * U * np.abs(prod)), (fp64, np.max(err / bound))


def _decaying():
    """5-point M-matrix, 28 x 28, diagonal 4 + 10, right-hand side e_1: x falls by 1e-40
    and more, and every entry of L and x is a sum of terms of one sign."""
    p = gridgen.laplacian_2d_dirichlet(28, shift=10.0)
    b = np.zeros((p.n, 1))
    b[0] = 1.0
    return p, b, oracle.reference(p, b)


def test_decaying_solution():
    """Entry by entry with FMAs (n u = 9e-14; 1e-11), against the largest entry otherwise."""
    p, b, ref = _decaying()
    xr = np.asarray(ref["x"]).reshape(-1)
    assert np.abs(xr).min() < 1e-30 * np.abs(xr).max()
    for fp64 in (0, 1):
        got = run(p, b, _opts(fp64))
        x = got["x"].reshape(-1)
        scale = np.abs(xr) if fp64 else np.abs(xr).max()
        assert np.max(np.abs(x - xr) / scale) <= 1e-11
        assert abs(got["logdet"] - ref["fac"].logdet()) <= 1e-12 * abs(ref["fac"].logdet())
        print("fp64_products=%d: worst relative error of an entry %.1e, of the largest %.1e"
              % (fp64, np.max(np.abs(x - xr) / np.abs(xr)), np.max(np.abs(x - xr)) / np.abs(xr).max()))


def test_option_keeps_the_fp64_kernels():
    """One launch a level where the tensor cores take two (operands split, tiles)."""
    from test_gpu_split import _arrow
    p = _arrow(129, 100)
    assert run(p, None, _opts(1))["stats"]["syrk"]["launches"] == 1
    assert run(p, None, _opts(0))["stats"]["syrk"]["launches"] == 2
