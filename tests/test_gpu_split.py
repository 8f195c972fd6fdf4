"""GPU parity of the binary64 updates on the tensor cores (bf16 slices).

Two leaf supernodes of s columns share one separator of b rows, so that a leaf's
panel takes trailing updates (s > 64), its update matrix has b rows and K = s,
and the separator takes trailing updates of its own. Sizes sit at the edges of
the 128 x 64 tiles, the 32-column blocks and the 64-column chunks.

Tolerances: the slices keep every entry of a row to 2^-64 of the row's largest,
so both this path and the oracle's FMAs are backward stable with a constant of a
few n u; the matrices have kappa < 100 after diagonal scaling, so entries agree
to well below the 1e-12 of the other binary64 parity tests.
"""
import numpy as np
import pytest

from gpu_util import check_parity, run
from helpers import lower_csc_from_dense
from lib_fixture import chol

pytestmark = pytest.mark.gpu


def _opts(mode=0, cap=0):
    o = chol().chol_default_options()
    o.small_max_cols = o.small_max_panel = 1   # everything wider than one column on the blocked path
    o.update_mode, o.device_mem_cap = mode, cap
    return o


def _arrow(s, b, spread=0, seed=0):
    """[D1 0 B1'; 0 D2 B2'; B1 B2 C], dense blocks, diagonally dominant; rows and
    columns scaled by powers of two within 2^+-spread."""
    rs = np.random.RandomState(1000 * s + b + seed)
    n = 2 * s + b
    A = rs.uniform(-1.0, 1.0, (n, n))
    A[s:2 * s, :s] = 0.0
    A = np.tril(A, -1) + np.tril(A, -1).T
    A[np.diag_indices(n)] = 1.05 * np.abs(A).sum(axis=1)
    if spread:
        d = np.ldexp(1.0, rs.randint(-spread, spread + 1, n))
        A = d[:, None] * A * d[None, :]
    cp, ri, vx = lower_csc_from_dense(A)
    return dict(n=n, colptr=cp, rowind=ri, values=vx, perm=np.arange(n, dtype=np.int32))


SIZES = [(2, 1), (31, 63), (32, 64), (33, 65), (64, 129), (65, 128), (96, 200), (127, 127), (128, 64), (129, 191),
         (257, 130), (300, 66)]


@pytest.mark.parametrize("s,b", SIZES)
@pytest.mark.parametrize("mode", [0, 1])
def test_tiles(s, b, mode):
    p = _arrow(s, b)
    rhs = np.random.RandomState(1).uniform(-1, 1, (p["n"], 2))
    got, _ = check_parity(p, rhs, _opts(mode))
    assert got["stats"]["syrk"]["launches"] >= 2   # operand split and tiles


@pytest.mark.parametrize("spread", [8, 200])
def test_power_of_two_scaling(spread):
    """Scaling rows and columns by powers of two changes no digit: L scales exactly."""
    p, q = _arrow(130, 100), _arrow(130, 100, spread)
    a, c = run(p, None, _opts()), run(q, None, _opts())
    d = np.sqrt(q["values"][q["colptr"][:-1]] / p["values"][p["colptr"][:-1]])
    lp, li, lx = a["L"]
    assert np.array_equal(c["L"][2], lx * d[li])


@pytest.mark.parametrize("mode", [0, 1])
def test_memory_cap_keeps_the_small_workspace_path(mode):
    p = _arrow(129, 100)
    got, ref = check_parity(p, None, _opts(mode, cap=1 << 40))
    assert got["stats"]["syrk"]["launches"] == 1
    check_parity(p, None, _opts(mode), ref=ref)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_not_finite(bad):
    """An entry of a leaf's off-diagonal rows spoils its row of the separator."""
    s, b = 70, 90
    p = _arrow(s, b)
    v = p["values"].copy()
    t = p["colptr"][3] + (s - 3) + 40          # column 3, row 40 of the separator
    assert p["rowind"][t] == 2 * s + 40
    v[t] = bad
    assert run(dict(p, values=v), None, _opts())["rc"] == 2 * s + 41


def test_not_positive_definite():
    p = _arrow(100, 80)
    v = p["values"].copy()
    v[p["colptr"][230]] = -1.0
    assert run(dict(p, values=v), None, _opts())["rc"] == 231


@pytest.mark.parametrize("s,b", [(33, 65), (64, 63), (65, 129), (130, 190), (257, 66)])
@pytest.mark.parametrize("mode", [0, 1])
def test_selected_inverse(s, b, mode):
    """The grouped products of the selected inverse (general, triangular and
    symmetric operands) against the dense inverse. kappa < 100 after scaling and
    n <= 580: entries within n u kappa < 1e-11 of the largest."""
    import torch
    P = chol()
    p = _arrow(s, b)
    rc, h = P.chol_analyze(p["n"], p["colptr"], p["rowind"], p["perm"], _opts(mode))
    assert rc == 0
    v = torch.as_tensor(p["values"], device="cuda")
    z = torch.empty_like(v)
    assert P.chol_factor(h, v) == 0 and P.chol_selected_inverse(h, z) == 0
    assert P.chol_check_waits(h) == 0
    P.chol_destroy(h)
    cols = np.repeat(np.arange(p["n"]), np.diff(p["colptr"]))
    A = np.zeros((p["n"], p["n"]))
    A[p["rowind"], cols] = p["values"]
    A = np.tril(A) + np.tril(A, -1).T
    ref = np.linalg.inv(A)[p["rowind"], cols]
    assert np.max(np.abs(z.cpu().numpy() - ref)) <= 1e-11 * np.max(np.abs(ref))


def test_selected_inverse_scaling():
    """Z scales exactly too: the K index of Z_RR U and U^T Z_RJ is balanced."""
    import torch
    P = chol()
    p = _arrow(130, 100)
    zs = []
    for q in (p, _arrow(130, 100, 60)):
        rc, h = P.chol_analyze(q["n"], q["colptr"], q["rowind"], q["perm"], _opts())
        v = torch.as_tensor(q["values"], device="cuda")
        z = torch.empty_like(v)
        assert rc == 0 and P.chol_factor(h, v) == 0 and P.chol_selected_inverse(h, z) == 0
        assert P.chol_check_waits(h) == 0
        P.chol_destroy(h)
        zs.append(z.cpu().numpy())
    d = np.sqrt(q["values"][q["colptr"][:-1]] / p["values"][p["colptr"][:-1]])
    cols = np.repeat(np.arange(p["n"]), np.diff(p["colptr"]))
    assert np.array_equal(zs[1], zs[0] / d[cols] / d[p["rowind"]])


# a level's panel entries times right-hand sides, 2 s b nrhs >= 8e6, nrhs >= 9, takes
# the tensor cores; 17 = a chunk of 16 and one right-hand side on the other path
@pytest.mark.parametrize("s,b,nrhs", [(300, 905, 16), (129, 2000, 17), (601, 1399, 9), (1030, 1030, 12)])
def test_solve_products(s, b, nrhs):
    """Solves of a system and of its scaling by powers of two, which is exactly the
    scaled solution; a column of NaN stays alone. n <= 3100, kappa < 100 after
    scaling: within n u kappa < 4e-11 of the largest entry."""
    import torch
    P = chol()
    rs = np.random.RandomState(7)
    x = rs.uniform(-1, 1, (2 * s + b, nrhs))
    got = []
    for spread in (0, 60):
        p = _arrow(s, b, spread)
        n, cols = p["n"], np.repeat(np.arange(p["n"]), np.diff(p["colptr"]))
        d = np.ones(n)
        if spread:
            d = np.sqrt(p["values"][p["colptr"][:-1]] / diag)
        diag = p["values"][p["colptr"][:-1]]
        if not spread:
            A = np.zeros((n, n))
            A[p["rowind"], cols] = p["values"]
            rhs = A @ x + np.tril(A, -1).T @ x
            rhs[:, nrhs - 1 if nrhs <= 16 else 3] = np.nan
        rc, h = P.chol_analyze(n, p["colptr"], p["rowind"], p["perm"], _opts())
        assert rc == 0 and P.chol_factor(h, torch.as_tensor(p["values"], device="cuda")) == 0
        y = torch.as_tensor(np.ascontiguousarray((rhs * d[:, None]).T), device="cuda")
        assert P.chol_solve(h, y, nrhs) == 0 and P.chol_check_waits(h) == 0
        P.chol_destroy(h)
        got.append(y.cpu().numpy().T * d[:, None])
    ok = ~np.isnan(rhs[0])
    assert np.max(np.abs(got[0][:, ok] - x[:, ok])) <= 4e-11
    assert np.isnan(got[0][:, ~ok]).all() and np.array_equal(got[0][:, ok], got[1][:, ok])


def test_solve_products_captured():
    """A solve captured before any other takes the binary64 kernels, one captured
    after a plain solve the tensor cores; both replay to the plain solve's x."""
    import torch
    P = chol()
    p = _arrow(300, 905)
    n, nrhs = p["n"], 16
    rc, h = P.chol_analyze(n, p["colptr"], p["rowind"], p["perm"], _opts())
    assert rc == 0 and P.chol_factor(h, torch.as_tensor(p["values"], device="cuda")) == 0
    b = torch.as_tensor(np.random.RandomState(2).uniform(-1, 1, (nrhs, n)), device="cuda")
    st = torch.cuda.Stream()
    got = []
    with torch.cuda.stream(st):
        one = b[0].clone()
        assert P.chol_solve(h, one, 1, st) == 0     # the workspaces every solve needs
        st.synchronize()
        for k in range(2):
            y = b.clone()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st, capture_error_mode="thread_local"):
                assert P.chol_solve(h, y, nrhs, st) == 0
            for _ in range(2):
                y.copy_(b)
                g.replay()
            st.synchronize()
            got.append(y.clone())
            x = b.clone()
            assert P.chol_solve(h, x, nrhs, st) == 0 and P.chol_check_waits(h, st) == 0
    P.chol_destroy(h)
    assert torch.equal(got[1], x)
    assert (got[0] - x).abs().max() <= 6e-11 * x.abs().max()


def test_selected_inverse_out_of_room():
    """A selected inverse that a memory cap refuses is refused again, wherever its
    allocations stop, and one that fits comes out as without a cap."""
    import torch
    P = chol()
    p = _arrow(130, 190)
    v = torch.as_tensor(p["values"], device="cuda")

    def attempt(cap):
        rc, h = P.chol_analyze(p["n"], p["colptr"], p["rowind"], p["perm"], _opts(cap=cap))
        assert rc == 0
        rcs, z = [P.chol_factor(h, v)], torch.empty_like(v)
        if rcs[0] == 0:
            rcs = [P.chol_selected_inverse(h, z) for _ in range(2)]
            assert P.chol_check_waits(h) == 0
        P.chol_destroy(h)
        return rcs, z
    want = attempt(1 << 40)
    assert want[0] == [0, 0]
    seen = set()
    for cap in np.linspace(1 << 18, 1 << 26, 256).astype(np.int64):
        rcs, z = attempt(int(cap))
        assert len(set(rcs)) == 1 and rcs[0] in (0, -1001)
        seen.add((len(rcs), rcs[0]))
        if rcs == [0, 0]:
            assert torch.equal(z, want[1])
    assert seen == {(1, -1001), (2, -1001), (2, 0)}


def test_factor_from_a_graph():
    """Blocked levels captured (the chain, bulk, side and small streams) and replayed."""
    p = _arrow(257, 130)
    o = _opts()
    o.use_graph = 1
    o.small_max_cols, o.small_max_panel = 64, 4096
    a, c = run(p, None, o), run(p, None, _opts())
    assert np.allclose(a["L"][2], c["L"][2], rtol=0, atol=1e-12 * np.abs(c["L"][2]).max())
    import torch
    P = chol()
    rc, h = P.chol_analyze(p["n"], p["colptr"], p["rowind"], p["perm"], o)
    v = torch.as_tensor(p["values"], device="cuda")
    for _ in range(3):
        assert P.chol_factor(h, v) == 0
    assert np.array_equal(P.chol_get_factor(h)[2], a["L"][2])
    P.chol_destroy(h)
