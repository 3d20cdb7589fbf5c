"""The order of the collected kNN candidates (csrc/knn.cu, warp_sort): every register count of the
sort, exact ties (lattices), nearly equal distances (a ring) and distances over more binades than
the sort's words tell apart, against the brute-force table, index by index."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1606_03135_gb300 import nodesets as NS
from paper_1606_03135_gb300 import rbffd as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def lattice(m, d):
    return np.stack(np.meshgrid(*[np.arange(m)] * d, indexing="ij"), -1).reshape(-1, d) / 8.0


def ring(k):
    t = 2 * np.pi * np.arange(k) / k
    r = 1.0 + 1e-9 * np.random.default_rng(k).standard_normal(k)
    return np.concatenate([[[0.0, 0.0]], np.stack([r * np.cos(t), r * np.sin(t)], 1)])


def powers():
    r = 2.0 ** -np.arange(0, 160, 0.5)  # squared distances over 320 binades
    t = 2.4 * np.arange(r.size)
    return np.stack([r * np.cos(t), r * np.sin(t)], 1)


SETS = {"lattice2d": lattice(24, 2), "lattice3d": lattice(9, 3), "ring": ring(230), "powers": powers(),
        "disk": NS.disk2d(1500, seed=2), "ball": NS.ball3d(1500, seed=2)}


@pytest.mark.parametrize("name", list(SETS))
@pytest.mark.parametrize("n", [2, 12, 31, 45, 64, 65, 96, 128])
def test_neighbours_are_in_the_exact_order(name, n):
    X = SETS[name]
    N, d = X.shape
    nbr_ref, d2_ref = O.knn(X, n)
    nbr = torch.zeros(N, n, dtype=torch.int32, device="cuda")
    rho2 = torch.zeros(N, dtype=torch.float64, device="cuda")
    ball = torch.zeros(N, dtype=torch.int32, device="cuda")
    rc = R.rbffd_stencils_noalloc(torch.from_numpy(X).cuda(), N, d, n, 0.5, nbr, rho2, ball)
    assert rc == 0
    assert np.array_equal(nbr.cpu().numpy(), nbr_ref)
    assert np.array_equal(rho2.cpu().numpy(), d2_ref[:, -1])
    assert np.array_equal(ball.cpu().numpy(), O.ball_len(d2_ref, 0.5))
