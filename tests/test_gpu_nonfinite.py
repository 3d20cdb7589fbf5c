"""Nodes that are not finite, or too far apart for their squared distances to be, are refused by
every entry point that searches stencils; the library works on afterwards."""
import numpy as np
import pytest

from paper_1606_03135_gb300 import nodesets as NS
from paper_1606_03135_gb300 import rbffd as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,ell", [(2, 13, 2), (3, 21, 2)])
@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf, -np.inf, 1e200, "scale"])
def test_nodes_without_distances_are_refused(d, n, ell, bad):
    X = NS.disk2d(3000, seed=2) if d == 2 else NS.ball3d(3000, seed=2)
    Y = X * 1e160 if bad == "scale" else X.copy()
    if bad != "scale":
        Y[1234, d - 1] = bad
    T = torch.from_numpy(Y).cuda()
    full = lambda v: np.full(len(X), v, np.int32)
    for make in (lambda: R.Plan(T, n, ell, 3, 0.5), lambda: R.Plan(Y, n, ell, 3, 1.0),
                 lambda: R.Plan(T, full(n), full(ell), full(3), 0.5),
                 lambda: R.Plan(T, n, ell, 3, 0.5, lebesgue_ref=R.LREF_CENTROID)):
        with pytest.raises(R.RbffdError) as e:
            make()
        assert e.value.code == R.EINVAL
    nbr = torch.empty(len(X), n, dtype=torch.int32, device="cuda")
    rho2 = torch.empty(len(X), dtype=torch.float64, device="cuda")
    ball = torch.empty(len(X), dtype=torch.int32, device="cuda")
    call = lambda t: R.rbffd_stencils_noalloc(t, len(X), d, n, 0.5, nbr, rho2, ball,
                                              torch.cuda.current_stream().cuda_stream)
    assert call(T) == R.EINVAL
    assert call(torch.from_numpy(X).cuda()) == R.OK
    with R.Plan(torch.from_numpy(X * 1e152).cuda(), n, ell, 3, 0.5) as p:  # far, but not too far
        p.assemble()
        assert np.isfinite(p.export_stencils()[1]).all()
