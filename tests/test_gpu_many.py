"""Forms that only levels of thousands of supernodes take: one warp a tiny
supernode in the factor, 8 or 16 lanes a supernode in the solves, the assembly of
a solve in two passes, and eight lanes a supernode in the logdet; and wide
one-CTA supernodes beside blocked ones.

A batch repeats a few small systems, so every copy must equal the first bit for
bit, the persistent kernel must give the same factor, and the same systems as a
small batch (other kernels) agree to rounding: n <= 300 and kappa < 1e4 give n u
kappa < 4e-10 at worst for x and n u < 1e-13 relative to a column for L; 1e-11
and 1e-12 are the other tests' bounds for such grids. Binary32: 1e-6 for L, and
kappa times the refinement's 1e-12 = 1e-8 for x.
"""
import numpy as np
import pytest

import gridgen
from gpu_util import check_parity, colmajor, to_dev
from helpers import lower_csc_from_dense
from lib_fixture import chol

pytestmark = pytest.mark.gpu


def _run(bd, b, precision=0, persistent=0):
    import torch
    P = chol()
    o = P.chol_default_options()
    o.precision, o.persistent = precision, persistent
    o.small_max_cols, o.small_max_panel, o.small_max_rows = 128, 16384, 512
    offs = bd["meta"]["offsets"].astype(np.int32)
    rc, h = P.chol_analyze_batch(len(offs) - 1, offs, bd["colptr"], bd["rowind"], bd["perm"], o)
    assert rc == 0 and P.chol_factor(h, to_dev(bd["values"])) == 0
    lx = P.chol_get_factor(h)[2]
    X = colmajor(b)
    if precision == 0:
        assert P.chol_solve(h, X, b.shape[1]) == 0
    else:
        assert P.chol_solve_refine(h, colmajor(b), X, b.shape[1], 1e-12, 50)[0] == 0
    torch.cuda.synchronize()
    rc, ld = P.chol_logdet_batch(h, len(offs) - 1)
    rc2, ld_all = P.chol_logdet(h)
    assert rc == 0 and rc2 == 0
    ns = P.chol_get_info(h).nsuper
    P.chol_destroy(h)
    return lx, X.cpu().numpy().reshape(b.shape, order="F"), np.asarray(ld), ld_all, ns


@pytest.mark.parametrize("precision,nrhs", [(0, 1), (0, 3), (1, 1)])
def test_many_copies(precision, nrhs):
    copies = 1013
    probs = gridgen.batch_2d(count=7, kmin=5, kmax=14, seed=3)
    one, many = gridgen.block_diagonal(probs), gridgen.block_diagonal(probs * copies)
    b = gridgen.rhs_uniform(one.n, nrhs, seed=5).reshape(one.n, nrhs)
    lx, x, ld, ld_all, ns = _run(many, np.tile(b, (copies, 1)), precision)
    assert ns > 32768
    lx = lx.reshape(copies, -1)
    x = x.reshape(copies, one.n, nrhs)
    ld = ld.reshape(copies, -1)
    for a in (lx, x, ld):
        assert np.array_equal(a, np.broadcast_to(a[0], a.shape))
    small = _run(one, b, precision)
    scale = 1.0 if precision == 0 else 1e6      # L is binary32 there
    assert np.max(np.abs(lx[0] - small[0])) <= 1e-12 * scale * np.max(np.abs(small[0]))
    assert np.max(np.abs(x[0] - small[1])) <= (1e-11 if precision == 0 else 1e-8) * np.max(np.abs(small[1]))
    assert np.max(np.abs(ld[0] - small[2])) <= 1e-12 * scale * np.max(np.abs(small[2]))
    assert abs(ld_all - copies * small[3]) <= 1e-12 * scale * abs(copies * small[3])
    if precision == 0:
        lp, xp, ldp, _, _ = _run(many, np.tile(b, (copies, 1)), 0, persistent=1)
        assert np.array_equal(lp, lx.ravel())


@pytest.mark.parametrize("s", [63, 64, 65, 100, 128])
@pytest.mark.parametrize("mode", [0, 1])
def test_wide_one_cta_beside_blocked(s, mode):
    """A leaf of s columns and 20 rows, which fits one CTA, beside one of 300 columns."""
    rs = np.random.RandomState(s)
    n, t, b = s + 300 + 20, 300, 20
    A = np.tril(rs.uniform(-1.0, 1.0, (n, n)), -1)
    A[s:s + t, :s] = 0.0
    A = A + A.T
    A[np.diag_indices(n)] = 1.05 * np.abs(A).sum(axis=1)
    cp, ri, vx = lower_csc_from_dense(A)
    o = chol().chol_default_options()
    o.small_max_cols, o.small_max_panel, o.small_max_rows, o.update_mode = 128, 20000, 512, mode
    p = dict(n=n, colptr=cp, rowind=ri, values=vx, perm=np.arange(n, dtype=np.int32))
    check_parity(p, rs.uniform(-1, 1, (n, 2)), o)


# rows of about 30, 240 and 1,200 entries (8 lanes; a warp a row); 66 right-hand
# sides pass the 64 that run side by side; 1,100 rows are 18 chunks of partials
@pytest.mark.parametrize("s,b,nrhs", [(15, 12, 1), (15, 11, 66), (120, 90, 3), (70, 1100, 3)])
def test_refinement_of_long_rows(s, b, nrhs):
    """Refined to a backward error of 1e-12 with kappa < 100 after scaling: x within 1e-9."""
    import torch
    P = chol()
    rs = np.random.RandomState(s + b)
    n = 2 * s + b
    A = np.tril(rs.uniform(-1.0, 1.0, (n, n)), -1)
    A[s:2 * s, :s] = 0.0
    A = A + A.T
    A[np.diag_indices(n)] = 1.05 * np.abs(A).sum(axis=1)
    cp, ri, vx = lower_csc_from_dense(A)
    o = P.chol_default_options()
    o.precision = P.CHOL_PREC_FP32
    o.small_max_cols = o.small_max_panel = 1
    rc, h = P.chol_analyze(n, cp, ri, np.arange(n, dtype=np.int32), o)
    assert rc == 0 and P.chol_factor(h, to_dev(vx)) == 0
    x = rs.uniform(-1, 1, (n, nrhs))
    X = colmajor(np.zeros((n, nrhs)))
    rc, iters, berr = P.chol_solve_refine(h, colmajor(A @ x), X, nrhs, 1e-12, 50)
    torch.cuda.synchronize()
    P.chol_destroy(h)
    assert rc == 0 and np.max(berr) <= 1e-12
    assert np.max(np.abs(X.cpu().numpy().reshape((n, nrhs), order="F") - x)) <= 1e-9
