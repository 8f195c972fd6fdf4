"""The framework's work as its users have it done, case by case: factor, solve, refine, differentiate.

Every case names a sparsity pattern (a grid stencil, an irregular graph or a
batch of grids), the analysis options a program would choose for it and the
calls it makes. `prepare` draws values and right-hand sides of that pattern from
a seed and analyzes the pattern; `run` makes the calls; `exact` solves the same
systems with plain torch in binary64.
"""
import functools
import math
import random

import numpy as np
import torch

import paper_2409_14009_gb300 as P
from paper_2409_14009_gb300.autograd import solve_logdet

DENSE_MAX = 14000          # largest order for which exact() forms the dense matrix
PRECISION = {"fp64": P.CHOL_PREC_FP64, "fp32": P.CHOL_PREC_FP32, "tf32": P.CHOL_PREC_TF32, "bf16": P.CHOL_PREC_BF16}


def listed():
    return [
        # the smallest problem that is factored in earnest: one 2D 5-point grid, default options, where
        # launches and the depth of the elimination tree are all that counts
        dict(name="2d64", call="factor_solve", grid="lap", dims="64x64", lo=0.1, hi=10.0, nrhs=1, prec="fp64", merge=0.0),
        # a 2D field solve on a ragged grid: a deep tree of narrow supernodes, many small levels
        dict(name="2d_301x423", call="factor_solve", grid="lap", dims="301x423", lo=0.1, hi=10.0, nrhs=1, prec="fp64", merge=0.1),
        # data in host memory, a small 3D box with three right-hand sides
        dict(name="host_3d_37x29x23", call="host", grid="lap", dims="37x29x23", lo=1e-2, hi=1e2, nrhs=3, prec="fp64", merge=0.1),
        # the benchmark's size: 3D 64^3 7-point, binary64 factor, 8 right-hand sides, log det
        dict(name="3d64", call="factor_solve", grid="lap", dims="64x64x64", lo=1e-2, hi=1e2, nrhs=8, prec="fp64", merge=0.1),
        # one factorization, many solves (time stepping, block methods): 16 right-hand sides on a kept factor
        dict(name="solve_3d48", call="solve", grid="lap", dims="48x48x48", lo=1e-2, hi=1e2, nrhs=16, prec="fp64", merge=0.1),
        # a matrix that comes without coordinates: ordered by the library's own nested dissection
        dict(name="irregular44", call="factor_solve", grid="irregular", dims="44x44x44", lo=0.1, hi=10.0, nrhs=1, prec="fp64", merge=0.1),
        # three degrees of freedom per node, 27-point, contrast 1e6: tensor-core updates, binary64 refinement
        dict(name="elast48_bf16", call="refine", grid="elast", dims="48x48x48", lo=1.0, hi=1e6, nrhs=1, prec="bf16", merge=0.1),
        # binary32 factor refined to binary64 accuracy, several right-hand sides, an odd box
        dict(name="refine_51x49x50", call="refine", grid="lap", dims="51x49x50", lo=1e-2, hi=1e2, nrhs=8, prec="fp32", merge=0.1),
        # a thousand small 2D systems of uneven sizes at once, binary64
        dict(name="batch1000", call="batch", grid="batch", dims="16..96", count=1000, lo=0.1, hi=10.0, nrhs=1, prec="fp64", merge=0.25),
        # the same in binary32 with refinement, as a program does that wants throughput
        dict(name="batch600_fp32", call="batch", grid="batch", dims="16..96", count=600, lo=0.1, hi=10.0, nrhs=1, prec="fp32", merge=0.25),
        # a differentiable solve: x and log det forward, gradients to b and to A's entries backward
        dict(name="grad_3d40", call="grad", grid="lap", dims="40x40x40", lo=1e-2, hi=1e2, nrhs=16, prec="fp64", merge=0.1),
        # the update without a workspace (RLB), vector problem, binary64
        dict(name="rlb_elast20", call="factor_solve", grid="elast", dims="20x20x20", lo=1.0, hi=1e6, nrhs=4, prec="fp64", merge=0.1, rlb=True),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(nodes_lo, nodes_hi, d, most):
        """An uneven d-dimensional box of about nodes_lo..nodes_hi nodes."""
        side = math.exp(rng.uniform(math.log(nodes_lo), math.log(nodes_hi)) / d)
        return "x".join(str(max(5, min(most, int(round(side * rng.uniform(0.8, 1.2)))))) for _ in range(d))

    nrhs = rng.choice([1, 1, 2, 3, 5, 8, 16])
    kind = rng.choice(["2d", "3d", "3d", "host", "solve", "irregular", "elast", "refine", "refine", "batch", "grad", "rlb"])
    if kind == "2d":
        return dict(call="factor_solve", grid="lap", dims=box(1000, 200000, 2, 460), lo=0.1, hi=10.0, nrhs=nrhs, prec="fp64", merge=rng.choice([0.0, 0.1]))
    if kind == "3d":
        return dict(call="factor_solve", grid="lap", dims=box(1000, 250000, 3, 64), lo=1e-2, hi=1e2, nrhs=nrhs, prec="fp64", merge=rng.choice([0.0, 0.1, 0.1]))
    if kind == "host":
        return dict(call="host", grid="lap", dims=box(1000, 60000, 3, 44), lo=1e-2, hi=1e2, nrhs=nrhs, prec="fp64", merge=0.1)
    if kind == "solve":
        return dict(call="solve", grid="lap", dims=box(4000, 110000, 3, 56), lo=1e-2, hi=1e2, nrhs=nrhs, prec="fp64", merge=0.1)
    if kind == "irregular":
        return dict(call="factor_solve", grid="irregular", dims=box(3000, 80000, 3, 48), lo=0.1, hi=10.0, nrhs=nrhs, prec="fp64", merge=0.1)
    if kind == "elast":
        return dict(call="refine", grid="elast", dims=box(1000, 50000, 3, 42), lo=1.0, hi=1e6, nrhs=rng.choice([1, 2, 4]), prec=rng.choice(["tf32", "bf16", "fp32"]), merge=0.1)
    if kind == "refine":
        return dict(call="refine", grid="lap", dims=box(1000, 150000, 3, 56), lo=1e-2, hi=1e2, nrhs=nrhs, prec="fp32", merge=0.1)
    if kind == "batch":
        return dict(call="batch", grid="batch", dims="16..%d" % rng.randint(40, 96), count=log_int(50, 800), lo=0.1, hi=10.0, nrhs=1, prec=rng.choice(["fp64", "fp32"]), merge=0.25)
    if kind == "grad":
        return dict(call="grad", grid="lap", dims=box(1000, 60000, 3, 42), lo=1e-2, hi=1e2, nrhs=nrhs, prec="fp64", merge=0.1)
    return dict(call="factor_solve", grid="elast", dims=box(500, 12000, 3, 24), lo=1.0, hi=1e6, nrhs=nrhs, prec="fp64", merge=0.1, rlb=True)


# ---- patterns ------------------------------------------------------------------

class Pattern:
    """Nodes, one stencil neighbour list per positive offset, and the lower CSC form."""


def _sides(case):
    return [int(v) for v in case["dims"].split("x")]


def _coords(dims):
    idx = np.arange(int(np.prod(dims)), dtype=np.int64)
    out, stride = [], 1
    for d in dims:
        out.append(idx // stride % d)
        stride *= d
    return idx, out


def _neighbours(dims, off):
    """Index of the node at `off` from each node, -1 outside the grid (axis 0 fastest)."""
    idx, co = _coords(dims)
    inside, shift, stride = np.ones(idx.size, bool), 0, 1
    for d, c, o in zip(dims, co, off):
        inside &= (c + o >= 0) & (c + o < d)
        shift += o * stride
        stride *= d
    return np.where(inside, idx + shift, -1)


def _dissection(dims):
    """Geometric nested dissection of a box grid (new -> old): the longest axis is split at its
    middle plane, low part, high part, plane; boxes of extent <= 2 lexicographically."""
    idx, co = _coords(dims)
    lo = [np.zeros(idx.size, np.int64) for _ in dims]
    hi = [np.full(idx.size, d, np.int64) for d in dims]
    key = np.zeros(idx.size, np.int64)
    live = np.ones(idx.size, bool)
    while True:
        ext = np.stack([h - l for l, h in zip(lo, hi)])
        split = live & (ext.max(0) > 2)
        axis = ext.argmax(0)
        key *= 4
        if not split.any():
            break
        for a in range(len(dims)):
            m = split & (axis == a)
            mid = lo[a] + ext[a] // 2
            below, above, on = m & (co[a] < mid), m & (co[a] > mid), m & (co[a] == mid)
            key[above] += 1
            key[on] += 2
            hi[a] = np.where(below, mid, hi[a])
            lo[a] = np.where(above, mid + 1, lo[a])
            live &= ~on
    lex = np.zeros(idx.size, np.int64)
    for d, c in zip(dims, co):
        lex = lex * d + c
    return np.lexsort((lex, key))


@functools.lru_cache(maxsize=12)
def _pattern(grid, dims, count):
    p = Pattern()
    if grid == "batch":
        lo, hi = (int(v) for v in dims.split(".."))
        rng = random.Random(count)
        sides = [rng.randint(lo, hi) for _ in range(count)]
        one = {k: (_neighbours((k, k), (1, 0)), _neighbours((k, k), (0, 1)), _dissection((k, k))) for k in set(sides)}
        p.sys_ptr = np.concatenate([[0], np.cumsum([k * k for k in sides])]).astype(np.int32)
        nb = [np.concatenate([np.where(one[k][o] >= 0, one[k][o] + b, -1) for k, b in zip(sides, p.sys_ptr)]) for o in (0, 1)]
        perm = np.concatenate([one[k][2] + b for k, b in zip(sides, p.sys_ptr)])
        p.units = None
    else:
        box = tuple(int(v) for v in dims.split("x"))
        if grid == "lap":
            offs = [tuple(int(a == b) for b in range(len(box))) for a in range(len(box))]
        else:
            offs = [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1) if (z, y, x) > (0, 0, 0)]
        nb = [_neighbours(box, o) for o in offs]
        p.units = None
        if grid == "elast":
            u = np.array(offs, float)
            u /= np.linalg.norm(u, axis=1, keepdims=True)
            p.units = np.eye(3)[None] + u[:, :, None] * u[:, None, :]
        if grid == "irregular":
            r = np.random.default_rng(12)
            nb = [np.where(r.random(b.size) < 0.35, b, -1) for b in nb]
        perm = None if grid == "irregular" else _dissection(box)
    p.nodes = nb[0].size
    p.dof = 1 if p.units is None else 3
    p.n = p.nodes * p.dof
    p.nb = [torch.as_tensor(b).cuda() for b in nb]
    # the node on the other side: pv[nb[i]] = i
    p.pv = []
    for b in nb:
        v = np.full(p.nodes, -1, np.int64)
        v[b[b >= 0]] = np.nonzero(b >= 0)[0]
        p.pv.append(torch.as_tensor(v).cuda())
    # the stored entries in the order in which _values lists them, then sorted to lower CSC
    node = torch.arange(p.nodes, device="cuda")
    rows, cols = [], []
    for a in range(p.dof):
        for b in range(a + 1):
            rows.append(node * p.dof + a)
            cols.append(node * p.dof + b)
    p.sel = []
    for b in p.nb:
        e = torch.nonzero(b >= 0).reshape(-1)
        p.sel.append(e)
        for a in range(p.dof):
            for c in range(p.dof):
                rows.append(b[e] * p.dof + a)
                cols.append(e * p.dof + c)
    rows, cols = torch.cat(rows), torch.cat(cols)
    _, p.order = torch.sort(cols * p.n + rows)
    p.rows, p.cols = rows[p.order], cols[p.order]
    p.rowind = p.rows.to(torch.int32).cpu().numpy()
    p.colptr = np.concatenate([[0], np.cumsum(torch.bincount(p.cols, minlength=p.n).cpu().numpy())]).astype(np.int64)
    if perm is None:
        rc, perm = P.chol_order_nd(p.n, p.colptr, p.rowind)
        if rc:
            raise P.CholError(rc, "chol_order_nd")
    elif p.dof > 1:
        perm = (perm[:, None] * p.dof + np.arange(p.dof)[None, :]).reshape(-1)
    p.perm = np.ascontiguousarray(perm, np.int32)
    return p


def _pattern_of(case):
    return _pattern(case["grid"], case["dims"], int(case.get("count", 0)))


def _values(p, case, g):
    """Entries of A: log-uniform edge weights; an edge that leaves a grid is a Dirichlet ghost (its
    weight counts on the diagonal only), an irregular graph has a small shift instead."""
    span = math.log(case["hi"] / case["lo"])

    def weights():
        return case["lo"] * torch.exp(span * torch.rand(p.nodes, generator=g, dtype=torch.float64, device="cuda"))

    ghosts = case["grid"] != "irregular"
    diag = [torch.zeros(p.nodes, dtype=torch.float64, device="cuda") for _ in range(p.dof * p.dof)]
    if not ghosts:
        diag[0] += 1e-2
    off = []
    for o, (nb, pv, e) in enumerate(zip(p.nb, p.pv, p.sel)):
        w, w2 = weights(), weights()
        up = w if ghosts else torch.where(nb >= 0, w, torch.zeros_like(w))
        down = torch.where(pv >= 0, w[pv.clamp(min=0)], w2 if ghosts else torch.zeros_like(w))
        for a in range(p.dof):
            for c in range(p.dof):
                k = 1.0 if p.units is None else float(p.units[o, a, c])
                diag[a * p.dof + c] += k * (up + down)
                off.append(-k * w[e])
    v = torch.cat([diag[a * p.dof + b] for a in range(p.dof) for b in range(a + 1)] + off)
    return v[p.order].contiguous()


def _inputs(case, seed):
    p = _pattern_of(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    values = _values(p, case, g)
    b = torch.rand((case["nrhs"], p.n), generator=g, dtype=torch.float64, device="cuda").mul_(2).sub_(1).t()
    w = torch.randn((case["nrhs"], p.n), generator=g, dtype=torch.float64, device="cuda").t() if case["call"] == "grad" else None
    return p, values, b, w


def _options(case):
    o = P.chol_default_options()
    o.precision = PRECISION[case["prec"]]
    o.merge_growth = case["merge"]
    if case.get("rlb"):
        o.update_mode = P.CHOL_UPDATE_RLB
    if case["call"] == "batch" and case["prec"] == "fp64":   # what chol_tune_batch finds for such batches
        o.small_max_cols, o.small_max_panel, o.small_max_rows = 128, 16384, 256
    return o


# ---- the calls -----------------------------------------------------------------

class Batch:
    """A program's handle of a batch: destroyed with it."""

    def __init__(self, p, options):
        rc, self.h = P.chol_analyze_batch(len(p.sys_ptr) - 1, p.sys_ptr, p.colptr, p.rowind, p.perm, options)
        if rc:
            raise P.CholError(rc, "chol_analyze_batch")
        self.count = len(p.sys_ptr) - 1

    def __del__(self):
        if getattr(self, "h", None):
            P.chol_destroy(self.h)
            self.h = None


def prepare(case, seed):
    p, values, b, w = _inputs(case, seed)
    s = dict(case=case, values=values, b=b, w=w)
    if case["call"] == "batch":
        s["solver"] = Batch(p, _options(case))
        return s
    s["solver"] = P.SparseCholesky(p.n, p.colptr, p.rowind, p.perm, _options(case))
    if case["call"] == "solve":
        s["solver"].factor(values)
    if case["call"] == "host":
        s["values"] = values.cpu().pin_memory()
        s["b"] = b.t().contiguous().cpu().pin_memory()      # n x nrhs column-major
        s["x"] = torch.empty_like(s["b"]).pin_memory()
    if case["call"] == "grad":
        s["values"] = values.requires_grad_(True)
        s["b"] = b.detach().requires_grad_(True)
    return s


def _ok(rc, where):
    if rc:
        raise P.CholError(rc, where)


def run(state):
    case, S, values, b = state["case"], state["solver"], state["values"], state["b"]
    call = case["call"]
    if call == "factor_solve":
        S.factor(values)
        return dict(x=S.solve(b), logdet=S.logdet())
    if call == "solve":
        return dict(x=S.solve(b))
    if call == "host":
        x = state["x"]
        rc, ld = P.chol_factor_solve_host(S.h, values, b, x, case["nrhs"], True, torch.cuda.current_stream())
        _ok(rc, "chol_factor_solve_host")
        return dict(x=x, logdet=ld)
    if call == "refine":
        S.factor(values)
        x = torch.empty_like(b)
        rc, _, _ = P.chol_solve_refine(S.h, b, x, case["nrhs"], 1e-14, 200, torch.cuda.current_stream())
        _ok(rc, "chol_solve_refine")
        return dict(x=x)
    if call == "batch":
        st = torch.cuda.current_stream()
        _ok(P.chol_factor_batch(S.h, values, st), "chol_factor_batch")
        if case["prec"] == "fp64":
            x = torch.empty_like(b).copy_(b)
            _ok(P.chol_solve_batch(S.h, x, case["nrhs"], st), "chol_solve_batch")
        else:
            x = torch.empty_like(b)
            rc, _, _ = P.chol_solve_refine(S.h, b, x, case["nrhs"], 1e-14, 200, st)
            _ok(rc, "chol_solve_refine")
        if case["prec"] != "fp64":
            return dict(x=x)
        rc, ld = P.chol_logdet_batch(S.h, S.count, st)
        _ok(rc, "chol_logdet_batch")
        return dict(x=x, logdet=ld)
    # a training step's loss: sum_k w_k^T x_k + log det A
    x, ld = solve_logdet(values, b, S)
    loss = (x * state["w"]).sum() + ld
    gv, gb = torch.autograd.grad(loss, (values, b))
    return dict(x=x.detach(), logdet=ld.detach(), grad_values=gv, grad_b=gb)


# ---- what a pass cannot do without ----------------------------------------------

@functools.lru_cache(maxsize=64)
def _symbolic(grid, dims, count):
    """(entries of L, sum of squared column counts) of the ordered pattern, without merging."""
    p = _pattern(grid, dims, count)
    rc, h = P.chol_analyze(p.n, p.colptr, p.rowind, p.perm, None)
    _ok(rc, "chol_analyze")
    info = P.chol_get_info(h)
    P.chol_destroy(h)
    return int(info.nnz_l), float(info.flops), len(p.rowind), p.n


def work(case):
    nnz_l, flops, nnz_a, n = _symbolic(case["grid"], case["dims"], int(case.get("count", 0)))
    solve = 4.0 * nnz_l * case["nrhs"]
    rhs = 16.0 * n * case["nrhs"]
    if case["call"] == "solve":       # the factor is read, from right to left again
        return dict(bytes=2 * 8.0 * nnz_l + rhs, flops=solve)
    if case["call"] == "grad":        # the selected inverse is twice the factor's work
        return dict(bytes=16.0 * nnz_a + 2 * rhs, flops=3 * flops + 2 * solve)
    return dict(bytes=8.0 * nnz_a + rhs, flops=flops + solve)


# ---- plain torch in 64 bits ------------------------------------------------------

def _solve_plain(p, values, b):
    """Conjugate gradients with a diagonal preconditioner, restarted on the true residual."""
    low = p.rows != p.cols
    r = torch.cat([p.rows, p.cols[low]])
    c = torch.cat([p.cols, p.rows[low]])
    v = torch.cat([values, values[low]])
    _, o = torch.sort(r * p.n + c)
    crow = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), torch.cumsum(torch.bincount(r, minlength=p.n), 0)])
    A = torch.sparse_csr_tensor(crow, c[o], v[o], size=(p.n, p.n))
    inv = (1.0 / values[~low]).unsqueeze(1)
    x = torch.zeros_like(b)
    for _ in range(4):
        res = b - A @ x
        d, z = torch.zeros_like(b), inv * res
        q, rz = z.clone(), (res * z).sum(0)
        goal = rz * 1e-26
        for it in range(6000):
            Aq = A @ q
            alpha = rz / (q * Aq).sum(0).clamp(min=1e-300)
            d += alpha * q
            res -= alpha * Aq
            z = inv * res
            new = (res * z).sum(0)
            if it % 50 == 0 and bool((new <= goal).all()):
                break
            q = z + (new / rz.clamp(min=1e-300)) * q
            rz = new
        x += d
    return x


def exact(case, seed):
    p, values, b, w = _inputs(case, seed)
    b = b.contiguous()
    out = {}
    if p.n <= DENSE_MAX:
        A = torch.zeros((p.n, p.n), dtype=torch.float64, device="cuda")
        A[p.rows, p.cols] = values
        A = torch.tril(A) + torch.tril(A, -1).t()
        C = torch.linalg.cholesky(A)

        def solve(v):
            x = torch.cholesky_solve(v, C)
            return x + torch.cholesky_solve(v - A @ x, C)

        out["x"] = solve(b)
        if case["call"] not in ("solve", "refine"):
            out["logdet"] = 2.0 * torch.log(torch.diagonal(C)).sum()
        if case["call"] == "grad":
            out["grad_b"] = solve(w)
            Z = torch.cholesky_inverse(C)
            twice = 1.0 + (p.rows != p.cols).to(torch.float64)
            outer = (out["grad_b"][p.rows] * out["x"][p.cols] + out["grad_b"][p.cols] * out["x"][p.rows]).sum(1) / 2
            out["grad_values"] = twice * (Z[p.rows, p.cols] - outer)
    else:
        out["x"] = _solve_plain(p, values, b)
        if case["call"] not in ("solve", "refine"):
            out["logdet"] = None
        if case["call"] == "grad":
            out["grad_b"] = _solve_plain(p, values, w.contiguous())
            out["grad_values"] = None
    if case["call"] == "host":
        out["x"] = out["x"].t().contiguous()
    if case["call"] == "batch":
        out.pop("logdet", None)
    return out
