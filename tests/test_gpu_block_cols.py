"""Binary64 parity for column blocks that are not multiples of a TRSM task's 16
rows, on levels with more blocked supernodes than the GPU holds CTAs at once (the
tasks of a launch then run one after another, so a row that two of them solve
would be solved twice).
"""
import functools

import pytest

import gridgen
import oracle
from gpu_util import check_parity
from lib_fixture import chol

pytestmark = pytest.mark.gpu


@functools.lru_cache(None)
def _case():
    p = gridgen.laplacian_neumann_varcoef((20, 20, 20), 1e-2, 1e2, 1e-6, seed=11)
    b = gridgen.rhs_uniform(p.n, 2, seed=11)
    return p, b, oracle.reference(p, b)


@pytest.mark.parametrize("block_cols", [8, 24, 40, 60, 63])
@pytest.mark.parametrize("mode", ["CHOL_UPDATE_RL", "CHOL_UPDATE_RLB"])
def test_block_cols_parity(block_cols, mode):
    p, b, ref = _case()
    P = chol()
    o = P.chol_default_options()
    o.block_cols, o.update_mode = block_cols, getattr(P, mode)
    o.small_max_cols = 1          # hundreds of blocked supernodes in the lower levels
    # kappa ~ 1e8: entries agree to kappa u; residual and backward error carry 1e-12
    check_parity(p, b, o, L_tol=1e-6, x_tol=1e-6, ref=ref)
