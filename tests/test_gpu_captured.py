"""Calls captured in a CUDA graph beside plain calls on the same handle."""
import numpy as np
import pytest

from lib_fixture import chol
from test_gpu_split import _arrow, _opts

pytestmark = pytest.mark.gpu


def _factored(p, scale=1.0):
    import torch
    P = chol()
    rc, h = P.chol_analyze(p["n"], p["colptr"], p["rowind"], p["perm"], _opts())
    v = torch.as_tensor(p["values"] * scale, device="cuda")
    assert rc == 0 and P.chol_factor(h, v) == 0
    return P, h, v


def test_selected_inverse_captured_is_not_yet_computed():
    """A captured selected inverse computes nothing before its replay: a plain call in
    between computes its own, and the replay computes it again. A is scaled by 4 in
    between, so that Z is exactly a quarter."""
    import torch
    p = _arrow(70, 90)
    P, h, v = _factored(p)
    st = torch.cuda.Stream()
    try:
        with torch.cuda.stream(st):
            z1, z2, zc = (torch.empty_like(v) for _ in range(3))
            assert P.chol_selected_inverse(h, z1, st) == 0     # the plan
            st.synchronize()
            assert P.chol_factor(h, 4.0 * v, st) == 0
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st, capture_error_mode="thread_local"):
                assert P.chol_selected_inverse(h, zc, st) == 0
            assert P.chol_selected_inverse(h, z2, st) == 0     # before any replay
            assert P.chol_check_waits(h, st) == 0
            assert torch.equal(z2, z1 / 4)
            assert P.chol_factor(h, 16.0 * v, st) == 0
            g.replay()
            assert P.chol_check_waits(h, st) == 0
            assert torch.equal(zc, z1 / 16)
            # captured while the plain call's Z is at hand, replayed after another factor
            assert P.chol_selected_inverse(h, z2, st) == 0
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st, capture_error_mode="thread_local"):
                assert P.chol_selected_inverse(h, zc, st) == 0
            assert P.chol_factor(h, v, st) == 0
            g.replay()
            assert P.chol_check_waits(h, st) == 0
            assert torch.equal(z2, z1 / 16) and torch.equal(zc, z1)
    finally:
        P.chol_destroy(h)
