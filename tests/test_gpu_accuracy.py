"""Accuracy of the null-space solves on ordinary node sets, against a double-double solve, next to
the oracle's partial-pivot LU.  Both are bound by the same rounding of the squared distances; what a
solver adds of its own shows in the medians.  Over 120 rows, with errors spread by a factor of two
about the median and half of them shared, two equally accurate solvers' medians agree to about 10%
(one standard deviation), so 1.25 is the line."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1606_03135_gb300 import nodesets as NS
from paper_1606_03135_gb300 import rbffd as R
from tests.test_gpu_degenerate import lattice
from tests.test_gpu_flat import errors
from tests.test_gpu_nullspace import check
from tests.test_gpu_parity import gpu_run

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,n,ell,m", [
    ("disk", 13, 2, 3), ("disk", 13, 2, 5), ("disk", 26, 3, 7), ("disk", 31, 4, 7), ("lattice", 31, 4, 7),
    ("ball", 21, 2, 5), ("ball", 45, 3, 7), ("ball", 71, 4, 7), ("ball", 113, 5, 7)])
def test_the_median_error_is_an_lu_solver_s(name, n, ell, m):
    X = (lattice(30, 2) if name == "lattice" else
         NS.disk2d(1500, seed=43) if name == "disk" else NS.ball3d(1500, seed=43))
    g = gpu_run(X, n, ell, m, 1.0)
    ref = O.assemble(X, n, ell, m, 1.0, R.STAB_SEQ)
    rows = np.random.default_rng(5).choice(len(X), 120, replace=False)
    e_gpu, e_ora = errors(X, g, ref, ell, m, rows, n)
    assert np.median(e_gpu) <= 1.25 * np.median(e_ora), (np.median(e_gpu), np.median(e_ora))


@pytest.mark.parametrize("d,n,ell,m,delta", [(2, 15, 1, 3, 0.3), (2, 16, 1, 3, 0.3), (3, 20, 1, 3, 0.3),
                                             (3, 21, 1, 3, 0.3), (3, 105, 4, 7, 0.03), (3, 105, 4, 7, 0.4)])
def test_shapes_on_both_sides_of_the_layout_rule(d, n, ell, m, delta):
    check(NS.jittered_grid(14 if d == 2 else 7, d, amp=0.3, seed=n), n, ell, m, delta)
