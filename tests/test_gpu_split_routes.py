"""Which binary64 products take the tensor cores, by the launches counted: a solve's
panel products take three launches a level and direction there (operands split,
right-hand sides split, tiles) and one on the FP64 pipe; a group of the selected
inverse's products two (operands, tiles) and one, or two with a reduction. And the
accuracy of solves that do take them.

In these matrices a leaf of s columns and b off-diagonal rows is level 0 (the other
leaf is one supernode with the separator): s b products a right-hand side; a level
of at least 8e6 products and 9 right-hand sides goes to the tensor cores.
"""
import numpy as np
import pytest

import test_gpu_split as split
from gpu_util import to_dev
from lib_fixture import chol

pytestmark = pytest.mark.gpu


def _stats(p, o, call):
    P = chol()
    rc, h = P.chol_analyze(p["n"], p["colptr"], p["rowind"], p["perm"], o)
    assert rc == 0
    try:
        assert P.chol_factor(h, to_dev(p["values"])) == 0
        P.chol_get_stats(h, reset=True)
        assert call(P, h) == 0 and P.chol_check_waits(h) == 0
        return {k: v["launches"] for k, v in P.chol_get_stats(h).items()}, P.chol_get_info(h).tc_products
    finally:
        P.chol_destroy(h)


@pytest.mark.parametrize("s,b,nrhs,want", [(500, 1000, 16, 3), (500, 999, 16, 1), (1000, 1000, 9, 3),
                                           (1000, 1000, 8, 1), (500, 1000, 17, 3 + 1), (500, 1000, 32, 3 + 3)])
def test_solve_launches(s, b, nrhs, want):
    p = split._arrow(s, b)
    x = to_dev(np.ones((nrhs, p["n"])))
    st, route = _stats(p, split._opts(), lambda P, h: P.chol_solve(h, x, nrhs))
    assert (st["solve_gemv"], st["solve_bpanel"]) == (want, want)
    assert route == (3 if want >= 3 else 1)


@pytest.mark.parametrize("how", ["cap", "option"])
def test_solve_launches_without_slices(how):
    p = split._arrow(500, 1000)
    o = split._opts(cap=1 << 40 if how == "cap" else 0)
    o.fp64_products = how == "option"
    x = to_dev(np.ones((16, p["n"])))
    st, route = _stats(p, o, lambda P, h: P.chol_solve(h, x, 16))
    assert (st["solve_gemv"], st["solve_bpanel"], route) == (1, 1, 0)


@pytest.mark.parametrize("how", ["slices", "cap", "option"])
def test_selected_inverse_launches(how):
    """Five groups: L_RJ T, Z_RR U, T^T T and U^T Z_RJ of the leaf, T^T T of the root."""
    p = split._arrow(65, 129)
    o = split._opts(cap=1 << 40 if how == "cap" else 0)
    o.fp64_products = how == "option"
    z = to_dev(p["values"])
    st, route = _stats(p, o, lambda P, h: P.chol_selected_inverse(h, z))
    if how == "slices":
        assert (st["selinv_gemm"], route) == (10, 5)
    else:
        assert st["selinv_gemm"] < 10 and route == 0


# edges of the 128-row tiles, odd K, parts of a sum, 9 to 16 right-hand sides
@pytest.mark.parametrize("s,b,nrhs", [(500, 1000, 16), (257, 1950, 16), (1300, 513, 13), (640, 1024, 17), (1001, 1000, 9)])
def test_solve_products(s, b, nrhs):
    assert s * b * min(nrhs, 16) >= 8e6
    split.test_solve_products(s, b, nrhs)
