"""Infinite diagonal entries (nodes pinned by an infinite penalty): the pivot's root
is infinite and its reciprocal zero, so the column of L below it is zero, x is zero
there and elsewhere that of the system without the node, the selected inverse is
zero in its row, and log det is infinite (of its own system only in a batch).

The remaining systems have n <= 400 and kappa < 1e4: n u kappa < 5e-10; 1e-10 of
the largest entry as in the other tests of such grids.
"""
import numpy as np
import pytest

import gridgen
from gpu_util import colmajor, to_dev
from helpers import dense_from_lower
from lib_fixture import chol

pytestmark = pytest.mark.gpu

TOL = 1e-10


def _pinned(p, pins):
    v = np.array(p["values"])
    v[p["colptr"][pins]] = np.inf
    return v


def _dense(p):
    return dense_from_lower(p["n"], p["colptr"], p["rowind"], p["values"])


MODES = {
    "default": {},
    "blocked": dict(small_max_cols=1, small_max_panel=1),
    "rlb": dict(update_mode=1),
    "one_cta": dict(small_max_cols=128, small_max_panel=16384, small_max_rows=512),
    "persistent": dict(small_max_cols=128, small_max_panel=16384, small_max_rows=512, persistent=1),
}


@pytest.mark.parametrize("mode", sorted(MODES))
@pytest.mark.parametrize("nrhs", [1, 3])
def test_pinned_nodes(mode, nrhs):
    import torch
    P = chol()
    p = gridgen.laplacian_2d_dirichlet_weighted(20, gridgen.SplitMix64(9))
    n = p.n
    # leaves, separators and the root, alone and next to one another
    pins = p["perm"][[0, 7, n // 3, n // 2, n // 2 + 1, n - 15, n - 4, n - 1]]
    keep = np.setdiff1d(np.arange(n), pins)
    o = P.chol_default_options()
    for k, val in MODES[mode].items():
        setattr(o, k, val)
    b = gridgen.rhs_uniform(n, nrhs, seed=2).reshape(n, nrhs)
    v = to_dev(_pinned(p, pins))
    rc, h = P.chol_analyze(n, p["colptr"], p["rowind"], p["perm"], o)
    assert rc == 0
    try:
        assert P.chol_factor(h, v) == 0
        got = []
        for solve in (P.chol_solve, P.chol_solve_noalloc):
            X = colmajor(b)
            assert solve(h, X, nrhs) == 0 and P.chol_check_waits(h) == 0
            got.append(X.cpu().numpy().reshape(n, nrhs))
        z = torch.empty_like(v)
        assert P.chol_selected_inverse(h, z) == 0 and P.chol_check_waits(h) == 0
        rc, ld = P.chol_logdet(h)
        rcb, ldb = P.chol_logdet_batch(h, 1)
        assert rc == 0 and rcb == 0
    finally:
        P.chol_destroy(h)
    A = _dense(p)[np.ix_(keep, keep)]
    ref = np.zeros((n, nrhs))
    ref[keep] = np.linalg.solve(A, b[keep])
    for x in got:
        assert np.array_equal(x[pins], np.zeros((len(pins), nrhs)))
        assert np.max(np.abs(x - ref)) <= TOL * np.max(np.abs(ref))
    Z = np.zeros((n, n))
    Z[np.ix_(keep, keep)] = np.linalg.inv(A)
    zr = Z[p["rowind"], np.repeat(np.arange(n), np.diff(p["colptr"]))]
    assert np.max(np.abs(z.cpu().numpy() - zr)) <= TOL * np.max(np.abs(zr))
    assert ld == np.inf and ldb[0] == np.inf


def test_pinned_node_of_a_batch():
    """The forms that levels of thousands of supernodes take; the systems without a
    pinned node come out bit for bit as without the pinned ones beside them."""
    P = chol()
    copies = 1013
    probs = gridgen.batch_2d(count=7, kmin=5, kmax=14, seed=3)
    one, many = gridgen.block_diagonal(probs), gridgen.block_diagonal(probs * copies)
    offs1 = one["meta"]["offsets"].astype(np.int32)
    offs = many["meta"]["offsets"].astype(np.int32)
    q = 3                                       # the pinned system
    n3 = probs[q].n
    local = probs[q]["perm"][[0, n3 // 2, n3 - 1]]
    vals1 = _pinned(one, offs1[q] + local)
    b = gridgen.rhs_uniform(one.n, 1, seed=5).reshape(one.n, 1)
    out = []
    for vals in (one["values"], vals1):
        rc, h = P.chol_analyze_batch(len(offs) - 1, offs, many["colptr"], many["rowind"], many["perm"])
        assert rc == 0
        try:
            assert P.chol_factor_batch(h, to_dev(np.tile(vals, copies))) == 0
            X = colmajor(np.tile(b, (copies, 1)))
            assert P.chol_solve_batch(h, X, 1) == 0 and P.chol_check_waits(h) == 0
            rc, ld = P.chol_logdet_batch(h, len(offs) - 1)
            assert rc == 0
            out.append((X.cpu().numpy().reshape(copies, one.n), np.asarray(ld).reshape(copies, 7)))
        finally:
            P.chol_destroy(h)
    (x0, ld0), (x1, ld1) = out
    other = np.ones(one.n, bool)
    other[offs1[q]:offs1[q + 1]] = False
    assert np.array_equal(x1[:, other], x0[:, other])
    rest = np.arange(7) != q
    assert np.array_equal(ld1[:, rest], ld0[:, rest]) and (ld1[:, q] == np.inf).all()
    keep = np.setdiff1d(np.arange(n3), local)
    A = _dense(probs[q])[np.ix_(keep, keep)]
    ref = np.zeros(n3)
    ref[keep] = np.linalg.solve(A, b[offs1[q]:offs1[q + 1], 0][keep])
    got = x1[:, offs1[q]:offs1[q + 1]]
    assert np.array_equal(got, np.broadcast_to(got[0], got.shape))
    assert np.array_equal(got[0][local], np.zeros(3)) and np.max(np.abs(got[0] - ref)) <= TOL * np.max(np.abs(ref))
