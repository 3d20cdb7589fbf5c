"""y = L u (csrc/assemble.cu, k_spmv): four lanes per row, row lengths around the lanes' strides and
node counts around a block's 64 rows, against the sums in extended precision on the CPU."""
import numpy as np
import pytest

from paper_1606_03135_gb300 import nodesets as NS
from paper_1606_03135_gb300 import rbffd as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ell,m", [(6, 2, 3), (7, 2, 3), (15, 2, 3), (16, 2, 3), (17, 2, 3), (33, 3, 5)])
@pytest.mark.parametrize("N", [63, 64, 65, 200])
def test_apply_equals_the_rows_sums(n, ell, m, N):
    X = NS.disk2d(N, seed=n)
    u = np.random.default_rng(N).standard_normal(N)
    with R.Plan(torch.from_numpy(X).cuda(), n, ell, m, 0.5) as p:
        p.assemble()
        ut = torch.from_numpy(u).cuda()
        y = torch.full((N,), float("nan"), dtype=torch.float64, device="cuda")
        p.apply(ut, y)
        rp, col, val, _ = p.export()
        y = y.cpu().numpy()
    for i in range(N):
        t = val[rp[i]:rp[i + 1]].astype(np.longdouble) * u[col[rp[i]:rp[i + 1]]]
        # at most n roundings of partial sums that are no larger than sum |t|
        assert abs(y[i] - t.sum()) <= n * 2.0 ** -53 * np.abs(t).sum() * 1.01, i
