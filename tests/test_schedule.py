"""The host-side schedule, read from the handle without a GPU.

Kernels of one launch run in any order and at the same time, so the tasks of a
launch must write disjoint entries; these tests check that on the task lists.
"""
import ctypes as C
import functools
import os
import subprocess

import numpy as np
import pytest

import gridgen
from lib_fixture import ROOT, chol


@pytest.fixture(scope="module")
def view(tmp_path_factory):
    from paper_2409_14009_gb300 import build
    chol()
    out = str(tmp_path_factory.mktemp("view") / "view.so")
    cmd = [build.NVCC, "-O1", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-x", "c++", "-I", build.INC, "-I",
           build.CSRC, os.path.join(ROOT, "tests", "schedule_view.cpp"), "-o", out, "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = C.CDLL(out)
    L.view_trsm.argtypes = [C.c_void_p, C.c_void_p]
    L.view_trsm.restype = C.c_int64
    L.view_trsm_rows.restype = C.c_int32
    return L


@functools.lru_cache(None)
def _grid(m):
    return gridgen.laplacian_neumann_varcoef((m, m, m), 1e-2, 1e2, 1e-6, seed=3)


def _analyze(m, **opts):
    P, p = chol(), _grid(m)
    o = P.chol_default_options()
    for k, v in opts.items():
        setattr(o, k, v)
    rc, h = P.chol_analyze(p.n, p["colptr"], p["rowind"], p["perm"], o)
    assert rc == 0
    return P, h


@pytest.mark.parametrize("block_cols", [8, 16, 24, 31, 40, 56, 60, 63, 64])
@pytest.mark.parametrize("small", [1, 64])
def test_trsm_rows_belong_to_one_task(view, block_cols, small):
    """Every row below a diagonal block is solved by exactly one task of its step."""
    P, h = _analyze(12, block_cols=block_cols, small_max_cols=small)
    n = view.view_trsm(h, None)
    t = np.zeros((n, 5), np.int32)
    view.view_trsm(h, t.ctypes.data)
    P.chol_destroy(h)
    assert n > 0
    height = view.view_trsm_rows()
    count = {}
    for J, k0, r0, s, ln in t.tolist():
        c = count.setdefault((J, k0), np.zeros(ln, np.int32))
        c[r0:r0 + height] += 1                  # the kernel bounds its rows by the supernode's
    for (J, k0), c in count.items():
        s = t[t[:, 0] == J][0, 3]
        r1 = min(k0 + block_cols, s)
        assert (c[:r1] == 0).all() and (c[r1:] == 1).all(), (J, k0, c[r1:].max(initial=0))
