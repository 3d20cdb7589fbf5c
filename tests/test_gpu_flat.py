"""Thin stencils (strips, slabs, nearly planar clouds): the constraints' pivots of degree 2 to 5 get
far below one, down to 2^-58 here, where the fixed-point elimination of the null-space solves leaves
its range and the stencil is done again in FP64.  Only an exactly zero pivot is an error.

The rows are held to a double-double solve next to the oracle's partial-pivot LU.  Both solvers'
errors are the systems' condition times rounding, so their medians over a set's rows agree to a
factor of 2 and, single rows being luck, their largest to a factor of 10."""
import itertools

import numpy as np
import pytest

from oracle import oracle as O
from paper_1606_03135_gb300 import nodesets as NS
from paper_1606_03135_gb300 import rbffd as R
from tests.hp_reference import dd_weights
from tests.test_gpu_boundary import run_bc
from tests.test_gpu_parity import gpu_run

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def strip(N, asp):
    rng = np.random.default_rng(3)
    y = (rng.random(N) * 2 - 1) * asp * 15 / N
    return np.stack([np.linspace(0, 1, N), y], 1)[rng.permutation(N)].copy()


def planar(side, asp):
    rng = np.random.default_rng(4)
    X = NS.square2d(side * side, seed=4)
    return np.concatenate([X, (rng.random((side * side, 1)) * 2 - 1) * asp * 2 / side], 1).copy()


def smallest_pivot(X, idx, ell):
    """Of the constraints, by elimination with partial pivoting, in the stencil's scaled coordinates."""
    x = X[idx] - X[idx[0]]
    x /= np.sqrt((x ** 2).sum(1).max())
    d = X.shape[1]
    ex = sorted((a for a in itertools.product(range(ell + 1), repeat=d) if sum(a) <= ell), key=sum)
    P = np.stack([np.prod(x ** np.array(a), 1) for a in ex], 1)
    least = np.inf
    for k in range(len(ex)):
        p = k + np.abs(P[k:, k]).argmax()
        P[[k, p]] = P[[p, k]]
        least = min(least, abs(P[k, k]))
        P[k + 1:, k:] -= np.outer(P[k + 1:, k] / P[k, k], P[k, k:])
    return least


def errors(X, g, ref, ell, m, rows, n):
    e = []
    for i in rows:
        idx = ref["nbr"][ref["owner"][i]]
        w = dd_weights(X, idx, ell, m, X[i:i + 1])[:, 0][np.argsort(idx)]
        e.append([np.linalg.norm(v["val"].reshape(-1, n)[i] - w) / np.linalg.norm(w) for v in (g, ref)])
    return np.array(e).T


SETS = {"strip 1e-2": lambda: strip(600, 1e-2), "strip 3e-3": lambda: strip(600, 3e-3),
        "strip 1e-3": lambda: strip(600, 1e-3), "strip 1e-4": lambda: strip(600, 1e-4),
        "planar 0.03": lambda: planar(22, 0.03), "planar 1e-3": lambda: planar(22, 1e-3),
        "slab 6e-3": lambda: NS.ball3d(500, seed=3) * np.array([1.0, 1.0, 6e-3])}


@pytest.mark.parametrize("name,n,ell,m", [
    ("strip 1e-2", 31, 4, 7), ("strip 3e-3", 31, 4, 7), ("strip 1e-3", 21, 3, 7),
    ("strip 1e-4", 31, 4, 7), ("strip 1e-4", 13, 2, 3), ("planar 0.03", 71, 4, 7),
    ("planar 1e-3", 45, 3, 7), ("slab 6e-3", 113, 5, 7)])
def test_thin_stencils_are_as_accurate_as_an_lu_solve(name, n, ell, m):
    X = SETS[name]()
    g = gpu_run(X, n, ell, m, 1.0)
    assert g["stats"]["n_singular"] == 0 and np.isfinite(g["val"]).all()
    ref = O.assemble(X, n, ell, m, 1.0, R.STAB_SEQ)
    rows = np.random.default_rng(1).choice(len(X), 24, replace=False)
    assert max(smallest_pivot(X, ref["nbr"][i], ell) for i in rows) < 2.0 ** -12
    e_gpu, e_ora = errors(X, g, ref, ell, m, rows, n)
    assert np.median(e_gpu) <= 2.0 * np.median(e_ora) + 1e-13, (e_gpu, e_ora)
    assert e_gpu.max() <= 10.0 * e_ora.max(), (e_gpu, e_ora)


@pytest.mark.parametrize("name,n,ell,delta", [("strip 1e-3", 31, 4, 0.5), ("planar 1e-3", 45, 3, 0.5),
                                              ("slab 6e-3", 113, 5, 0.6)])
def test_thin_stencils_in_teams_and_chunks_are_bitwise_equal(name, n, ell, delta):
    X = SETS[name]()
    a = gpu_run(X, n, ell, 7, delta)
    assert a["stats"]["max_ball"] > 5 and np.isfinite(a["val"]).all()
    for kw in (dict(team=32), dict(team=64, rhs_chunk=3), dict(team=256), dict(team=512, rhs_chunk=5)) + \
            ((dict(team=96), dict(team=128, rhs_chunk=2)) if n < 100 else ()):
        b = gpu_run(X, n, ell, 7, delta, **kw)
        for key in ("row_ptr", "col", "val", "owner", "is_center", "lam_row"):
            assert np.array_equal(a[key], b[key]), (key, kw)


def test_normal_derivatives_of_thin_stencils():
    """The Neumann rows differ from the oracle's no more than both solvers' Laplacian rows of the
    same nodes are off (same matrices, so the same condition), up to a factor of 4."""
    X, n, ell, m = strip(600, 1e-3), 21, 3, 7
    lap = gpu_run(X, n, ell, m, 1.0)
    ref = O.assemble(X, n, ell, m, 1.0, R.STAB_SEQ)
    rows = np.random.default_rng(2).choice(len(X), 24, replace=False)
    e = errors(X, lap, ref, ell, m, rows, n).sum(0)
    bc, nrm = np.zeros(len(X), np.uint8), np.zeros_like(X)
    bc[rows] = 2
    nrm[rows] = [0.6, 0.8]
    g = run_bc(X, bc, nrm, n, ell, m, 1.0)
    r = O.assemble(X, n, ell, m, 1.0, R.STAB_SEQ, bc=bc, normals=nrm)
    a, b = (v["val"].reshape(-1, n)[rows] for v in (g, r))
    assert np.median(np.linalg.norm(a - b, axis=1) / np.linalg.norm(b, axis=1)) <= 4.0 * np.median(e)
