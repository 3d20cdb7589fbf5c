"""Neumann rows are linear in the normal, of any length: the oracle's rows at the method's 1e-9, and
for lengths a power of two apart the same bits."""
import numpy as np
import pytest

from paper_1606_03135_gb300 import nodesets as NS
from tests.test_gpu_boundary import compare_bc, run_bc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def ball_bc(N):
    X, bc, _ = NS.ball3d_bc(N, seed=5)
    nrm = X / np.maximum(np.linalg.norm(X, axis=1), 1e-12)[:, None]
    return X, np.where(bc > 0, 2, 0).astype(np.uint8), nrm


@pytest.mark.parametrize("d,n,ell,m", [(2, 12, 2, 3), (2, 13, 2, 5), (2, 31, 4, 7), (3, 21, 2, 3),
                                       (3, 45, 3, 7), (3, 71, 4, 7)])
@pytest.mark.parametrize("length", [1.0, 7.0, 20.0, 400.0, 1e12, 1e-9, 1e-100])
def test_rows_of_long_and_short_normals(d, n, ell, m, length):
    X, bc, nrm = NS.disk2d_bc(900, seed=1) if d == 2 else ball_bc(1200)
    compare_bc(X, bc, nrm * length, n, ell, m, 1.0)


@pytest.mark.parametrize("n,ell,m", [(12, 2, 3), (31, 4, 7)])
def test_lengths_a_power_of_two_apart_give_the_same_bits(n, ell, m):
    X, bc, nrm = NS.disk2d_bc(900, seed=1)
    a = run_bc(X, bc, nrm, n, ell, m, 0.5)
    b = bc > 0
    for e in (-300, -7, 1, 9, 300):
        g = run_bc(X, bc, np.ldexp(nrm, e), n, ell, m, 0.5)
        v, w = (r["val"].reshape(-1, n) for r in (a, g))
        assert np.array_equal(np.ldexp(v[b], e), w[b]) and np.array_equal(v[~b], w[~b])
        assert np.array_equal(np.ldexp(a["lam_row"][b], e), g["lam_row"][b])


def test_a_zero_normal_gives_a_zero_row():
    X, bc, nrm = NS.disk2d_bc(900, seed=1)
    k = np.flatnonzero(bc)[0]
    nrm[k] = 0.0
    g = run_bc(X, bc, nrm, 31, 4, 7, 1.0)
    assert np.all(g["val"].reshape(-1, 31)[k] == 0.0)
