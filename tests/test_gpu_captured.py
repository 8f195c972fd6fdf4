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


@pytest.mark.parametrize("capture_mode", ["thread_local", "global", "relaxed"])
def test_solve_route_does_not_depend_on_the_calls_before(capture_mode):
    """The first solve with many right-hand sides takes the tensor cores whether it is
    captured or not, and gives the same bits. (600 x 1000 panel entries, 16 right-hand
    sides: 9.6e6 products in level 0, more than the 8e6 from which a level goes there.)"""
    import torch
    p = _arrow(600, 1000)
    n, nrhs = p["n"], 16
    b = torch.as_tensor(np.random.RandomState(2).uniform(-1, 1, (nrhs, n)), device="cuda")
    P, plain, _ = _factored(p)
    _, h, _ = _factored(p)
    st = torch.cuda.Stream()
    try:
        x = b.clone()
        assert P.chol_get_info(plain).tc_products == 1
        assert P.chol_solve(plain, x, nrhs) == 0 and P.chol_check_waits(plain) == 0
        assert P.chol_get_info(plain).tc_products == 3
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            one = b[0].clone()
            assert P.chol_solve(h, one, 1, st) == 0        # the workspaces every solve needs
            st.synchronize()
            y = b.clone()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st, capture_error_mode=capture_mode):
                assert P.chol_solve(h, y, nrhs, st) == 0
            for _ in range(2):
                y.copy_(b)
                g.replay()
            assert P.chol_check_waits(h, st) == 0
            assert torch.equal(y, x)
            y.copy_(b)
            assert P.chol_solve(h, y, nrhs, st) == 0 and P.chol_check_waits(h, st) == 0
            assert torch.equal(y, x) and P.chol_get_info(h).tc_products == 3
    finally:
        P.chol_destroy(h)
        P.chol_destroy(plain)
