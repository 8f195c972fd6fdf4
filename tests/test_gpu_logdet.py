"""log det against the logarithms of the factor's own diagonal: only the logarithms
and their sum round."""
import math

import numpy as np
import pytest

from gpu_util import to_dev
from lib_fixture import chol

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [40, 40000])   # a warp or eight lanes a supernode
def test_near_one(n):
    """Roots a little above and below one: the log det of every 1 x 1 system keeps its
    relative accuracy (binary64 logarithms err by an ulp at most; a factor of 2)."""
    P = chol()
    k = np.arange(1, n + 1) % 1000 + 1
    root = 1.0 + np.where(np.arange(n) % 2, k, -k) * 2.0 ** -24    # roots' squares have at most 52 bits
    cp, ri = np.arange(n + 1, dtype=np.int64), np.arange(n, dtype=np.int32)
    rc, h = P.chol_analyze_batch(n, np.arange(n + 1, dtype=np.int32), cp, ri)
    assert rc == 0
    try:
        assert P.chol_factor_batch(h, to_dev(root * root)) == 0
        d = P.chol_get_factor(h)[2]
        assert np.max(np.abs(d - root)) <= 2.0 ** -52
        rc, ld = P.chol_logdet_batch(h, n)
        assert rc == 0
    finally:
        P.chol_destroy(h)
    ref = np.array([2.0 * math.log1p(r - 1.0) for r in d])
    assert np.max(np.abs(ld - ref) / np.abs(ref)) <= 4 * 2.0 ** -52
