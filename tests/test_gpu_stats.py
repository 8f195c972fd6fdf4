"""The launch statistics count every supernode's work once, whichever kernels
factor it."""
import gridgen
import pytest

from gpu_util import run, to_dev
from lib_fixture import chol

pytestmark = pytest.mark.gpu


def _work(p, **opts):
    o = chol().chol_default_options()
    for k, v in opts.items():
        setattr(o, k, v)
    got = run(p, None, o)
    assert got["rc"] == 0
    st, info = got["stats"], got["info"]
    return {k: st[k]["flops"] for k in ("small", "potrf", "trsm", "gemm", "syrk")}, info


def test_wide_one_cta_supernodes_beside_blocked_ones():
    """With supernodes beyond the one-CTA class, those of the class wider than 64
    columns take the blocked kernels: their work belongs there alone."""
    p = gridgen.laplacian_2d_dirichlet(160)
    wide = dict(small_max_panel=24576, small_max_rows=512)
    got, info = _work(p, small_max_cols=128, **wide)
    ref, ref_info = _work(p, small_max_cols=64, **wide)      # the same kernels
    assert info.n_small + info.n_large == info.nsuper_storage
    assert (info.n_small, info.n_large) == (ref_info.n_small, ref_info.n_large)
    assert ref_info.n_large > 2 and got == ref


def test_gather_launches():
    """The selected inverse gathers by the factor's assembly tasks, level by level in the
    same launches (one level has CTA-sized and warp-sized tasks, few enough for one)."""
    P = chol()
    p = gridgen.elasticity_27pt(10)
    rc, h = P.chol_analyze(p.n, p["colptr"], p["rowind"], p["perm"])
    assert rc == 0
    try:
        v = to_dev(p["values"])
        assert P.chol_factor(h, v) == 0 and P.chol_selected_inverse(h, to_dev(p["values"])) == 0
        assert P.chol_check_waits(h) == 0
        st = P.chol_get_stats(h)
    finally:
        P.chol_destroy(h)
    assert st["selinv_gather"]["launches"] == st["assemble"]["launches"] > 0
