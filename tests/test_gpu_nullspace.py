"""Null-space local solves (plans of one shape, degree 1 to 5, r^3 to r^7 with ell >= (m - 1) / 2) at
the edges of their shapes: n = M and M + 1 (no or one node beside the basic ones), odd and even M,
more other nodes than basic ones, K on both sides of the refinement size, the largest exponent the
degree allows, and one exponent or degree more (the saddle-point factorization).

Every row is held to the oracle at the method's 1e-9 of its largest weight; a row that misses it is
compared with a double-double solve instead, where it may be off by at most 1e-9 or twice the
oracle's own error, whichever is larger (the oracle's LU rounds too: at the condition numbers of
these shapes, up to 1e7, two FP64 solvers differ by about the sum of their errors)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1606_03135_gb300 import nodesets as NS
from paper_1606_03135_gb300 import rbffd as R
from tests.hp_reference import dd_weights
from tests.test_gpu_parity import gpu_run

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def check(X, n, ell, m, delta, mode=R.STAB_SEQ, **kw):
    g = gpu_run(X, n, ell, m, delta, mode, **kw)
    ref = O.assemble(X, n, ell, m, delta, mode)
    assert np.array_equal(g["owner"], ref["owner"]) and np.array_equal(g["col"], ref["col"])
    a, b = g["val"].reshape(-1, n), ref["val"].reshape(-1, n)
    err = np.abs(a - b).max(1) / np.abs(b).max(1)
    far = np.flatnonzero(err > 1e-9)
    assert far.size <= 0.02 * len(X)
    for i in far[:8]:
        idx = ref["nbr"][ref["owner"][i]]
        w = dd_weights(X, idx, ell, m, X[i:i + 1])[:, 0][np.argsort(idx)]
        e_gpu, e_ora = (np.abs(v[i] - w).max() / np.abs(w).max() for v in (a, b))
        assert e_gpu <= max(1e-9, 2.0 * e_ora), (i, e_gpu, e_ora)
    return g


@pytest.mark.parametrize("d,n,ell,m", [
    (2, 6, 2, 5), (2, 7, 2, 5), (2, 21, 5, 7), (2, 4, 1, 3),         # n = M, M + 1
    (2, 31, 4, 9), (2, 31, 4, 7), (2, 31, 3, 9),                     # m against 2 ell + 1 and 7
    (2, 90, 2, 3), (2, 93, 2, 5), (2, 94, 2, 5),                     # s >> M; K = 99, 100
    (3, 20, 3, 7), (3, 21, 3, 7), (3, 45, 3, 5), (3, 64, 4, 7),      # M = 20, 35; K = 99
    (3, 11, 2, 5), (3, 25, 2, 3), (3, 5, 1, 3)])
def test_shapes_at_delta_one(d, n, ell, m):
    check(NS.jittered_grid(14 if d == 2 else 6, d, amp=0.3, seed=n), n, ell, m, 1.0)


@pytest.mark.parametrize("d,n,ell,m,delta", [(2, 31, 4, 7, 0.15), (2, 90, 2, 3, 0.1),
                                             (3, 45, 3, 7, 0.15), (3, 64, 4, 7, 0.3)])
@pytest.mark.parametrize("kw", [{}, dict(team=32), dict(team=512), dict(team=96, rhs_chunk=1),
                                dict(team=256, rhs_chunk=7)])
def test_many_columns_in_teams_and_chunks_are_bitwise_equal(d, n, ell, m, delta, kw):
    X = NS.jittered_grid(20 if d == 2 else 8, d, seed=3)
    a = gpu_run(X, n, ell, m, delta)
    b = gpu_run(X, n, ell, m, delta, **kw)
    assert a["stats"]["max_ball"] > 15
    for key in ("row_ptr", "col", "val", "owner", "is_center", "lam_row"):
        assert np.array_equal(a[key], b[key]), key


@pytest.mark.parametrize("mode", [R.STAB_SEQ, R.STAB_OFF, R.STAB_FALLBACK])
@pytest.mark.parametrize("scale", [1e-30, 1.0, 1e30])
def test_modes_and_scales(mode, scale):
    check(NS.disk2d(700, seed=9) * scale, 21, 3, 7, 0.4, mode)


@pytest.mark.parametrize("d,n,ell,m,delta", [(3, 45, 3, 7, 0.5), (3, 64, 4, 7, 0.6), (2, 31, 4, 7, 0.5),
                                             (3, 71, 4, 7, 1.0), (3, 113, 5, 7, 0.5)])
def test_refining_every_system_works_in_every_team(d, n, ell, m, delta):
    """The refinement step, whole and chunked, in teams of every size; K >= 100 also as it comes."""
    X = NS.ball3d(600, seed=4) if d == 3 else NS.disk2d(900, seed=4)
    a = check(X, n, ell, m, delta, refine=R.REFINE_ALL)
    assert a["stats"]["flops_refine"] > 0
    for refine, a in ((R.REFINE_ALL, a), (R.REFINE_AUTO, check(X, n, ell, m, delta))):
        for kw in (dict(team=32), dict(team=64, rhs_chunk=3), dict(team=256), dict(team=512, rhs_chunk=5)):
            b = gpu_run(X, n, ell, m, delta, refine=refine, **kw)
            for key in ("row_ptr", "col", "val", "owner", "is_center", "lam_row"):
                assert np.array_equal(a[key], b[key]), (key, refine, kw)


def test_nearly_flat_stencils_match_the_lu_option():
    """Nodes of a thin slab: the constraints' pivots span four orders of magnitude, so B and
    the columns' constraint weights grow; the partial-pivot LU of the whole system (an independent
    path of the library) gives the same rows up to the conditioning of such stencils."""
    X = NS.jittered_grid(12, 2, amp=0.3, seed=5) * np.array([1.0, 1e-2])
    a = gpu_run(X, 12, 2, 3, 1.0)["val"].reshape(-1, 12)
    b = gpu_run(X, 12, 2, 3, 1.0, factor=R.FACTOR_LU)["val"].reshape(-1, 12)
    err = np.abs(a - b).max(1) / np.abs(b).max(1)
    assert err.max() < 1e-6 and np.median(err) < 1e-9
