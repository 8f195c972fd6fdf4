"""Lost waits of the tensor-core tiles of the binary64 products, made on purpose
without a fault: bits 2, 4 and 8 of chol_options.test_unreachable_flags make one
epilogue warp of every tile (of the factor, the solves' panel products, the
selected inverse) take its waits as run out at once. The other roles of the CTA,
whose own waits are met, have to leave with it; the call reports CHOL_ETIMEOUT and
the context stays usable.
"""
import numpy as np
import pytest

from gpu_util import to_dev
from lib_fixture import chol
from test_gpu_split import _arrow, _opts

pytestmark = pytest.mark.gpu


def _handle(p, flags, mode=0):
    P = chol()
    o = _opts(mode)
    o.test_unreachable_flags = flags
    rc, h = P.chol_analyze(p["n"], p["colptr"], p["rowind"], p["perm"], o)
    assert rc == 0
    return P, h


# one chunk a tile and one tile a CTA; several of both
@pytest.mark.parametrize("s,b", [(70, 90), (300, 1400)])
@pytest.mark.parametrize("mode", [0, 1])
def test_factor(s, b, mode):
    P, h = _handle(_arrow(s, b), 2, mode)
    v = to_dev(_arrow(s, b)["values"])
    try:
        for _ in range(2):
            # the broken updates may also show up as a pivot that is not positive
            rc = P.chol_factor(h, v)
            assert rc == P.CHOL_ETIMEOUT or rc > 0
            assert P.chol_solve(h, to_dev(np.ones(2 * s + b)), 1) == P.CHOL_ESTATE
    finally:
        P.chol_destroy(h)
    check = _handle(_arrow(s, b), 0, mode)[1]
    assert P.chol_factor(check, v) == 0 and P.chol_check_waits(check) == 0
    P.chol_destroy(check)


@pytest.mark.parametrize("s,b", [(65, 129), (300, 905)])
def test_selected_inverse(s, b):
    import torch
    p = _arrow(s, b)
    P, h = _handle(p, 8)
    v = to_dev(p["values"])
    try:
        assert P.chol_factor(h, v) == 0
        assert P.chol_selected_inverse(h, torch.empty_like(v)) == 0    # asynchronous
        assert P.chol_check_waits(h) == P.CHOL_ETIMEOUT
        assert P.chol_check_waits(h) == 0                              # the record was cleared
        assert P.chol_factor(h, v) == 0
    finally:
        P.chol_destroy(h)
