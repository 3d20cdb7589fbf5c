"""Stencils that the null space of the constraints cannot solve: lattices (at the edge of a lattice a
polynomial of the basis may vanish at every node of a stencil, so its constraints depend on each
other) and nodes nearer each other than rounding.  Plans of one shape
answer them as the saddle-point layout of the other plans does; a plan whose last node is one
smaller in degree and stencil size has that layout, and the same rows everywhere else."""
import itertools

import numpy as np
import pytest

from oracle import oracle as O
from paper_1606_03135_gb300 import nodesets as NS
from paper_1606_03135_gb300 import rbffd as R
from tests.test_gpu_parity import gpu_run, gpu_run_mixed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def lattice(side, d, h=0.1):
    g = np.arange(side) * h
    return np.stack(np.meshgrid(*[g] * d, indexing="ij"), -1).reshape(-1, d).copy()


def constraints(X, idx, ell):
    """Rank and consistency of P^T w = g (Laplacian at the center) by the singular values of P."""
    x = X[idx] - X[idx[0]]
    x /= np.sqrt((x ** 2).sum(1).max())
    ex = [a for a in itertools.product(range(ell + 1), repeat=X.shape[1]) if sum(a) <= ell]
    P = np.stack([np.prod(x ** np.array(a), 1) for a in ex], 1)
    g = np.array([2.0 * (sorted(a)[-1] == 2 and sum(a) == 2) for a in ex])
    U, s, Vt = np.linalg.svd(P)
    null = Vt[int((s > 1e-10 * s[0]).sum()):]
    return len(null), bool(np.abs(null @ g).max(initial=0.0) < 1e-9)


def saddle(X, n, ell, m, delta, mode=R.STAB_SEQ):
    """The rows from a plan of two shapes."""
    N = len(X)
    nn, ll = np.full(N, n, np.int32), np.full(N, ell, np.int32)
    nn[-1], ll[-1] = n - 1, ell - 1
    return gpu_run_mixed(X, nn, ll, np.full(N, m, np.int32), delta, mode)


CASES = [(2, 30, 16, 4, 7), (2, 30, 25, 4, 7), (3, 9, 27, 3, 7), (3, 10, 45, 3, 7), (3, 10, 21, 2, 3),
         (3, 10, 71, 4, 7), (3, 9, 113, 5, 7)]


@pytest.mark.parametrize("d,side,n,ell,m", CASES)
def test_lattices_are_solved_like_saddle_point_systems(d, side, n, ell, m):
    """Full rank: the rows of the two layouts within 1e-9 (condition 1e7 at most).  Dependent but
    consistent constraints have one solution, but which of two equal monomials takes the pivot is
    decided by rounding, and the multipliers grow to its inverse: the rows agree to sqrt(eps).
    Inconsistent ones have none; the row is finite, as from the saddle-point layout, and no larger
    than 100 times its largest."""
    X = lattice(side, d)
    N = len(X)
    g = gpu_run(X, n, ell, m, 1.0)
    ref = saddle(X, n, ell, m, 1.0)
    assert g["stats"]["n_singular"] == 0
    kind = np.array([constraints(X, g["nbr"][i], ell) for i in range(N)])
    full = kind[:, 0] == 0
    some = ~full & (kind[:, 1] == 1)
    assert (~full).sum() > 0
    a = g["val"].reshape(N, n)[:-1]
    b = np.array([ref["val"][ref["row_ptr"][i]:ref["row_ptr"][i + 1]] for i in range(N - 1)])
    full, some = full[:-1], some[:-1]
    err = np.linalg.norm(a - b, axis=1) / np.linalg.norm(b, axis=1)
    assert np.isfinite(a).all()
    assert not full.any() or err[full].max() < 1e-9
    assert not some.any() or err[some].max() < 2e-8
    assert np.abs(a).max() <= 100.0 * np.abs(b).max()


@pytest.mark.parametrize("d,side,n,ell,delta", [(2, 30, 25, 4, 0.4), (3, 9, 45, 3, 0.3), (3, 8, 64, 4, 0.5)])
def test_lattices_in_teams_and_chunks_are_bitwise_equal(d, side, n, ell, delta):
    X = lattice(side, d)
    for mode in (R.STAB_OFF, R.STAB_FALLBACK):
        a = gpu_run(X, n, ell, 7, delta, mode)
        assert a["stats"]["max_ball"] > 5 and a["stats"]["n_singular"] == 0
        for kw in (dict(team=32), dict(team=64, rhs_chunk=3), dict(team=256), dict(team=512, rhs_chunk=5),
                   dict(max_ctas=1500)):
            b = gpu_run(X, n, ell, 7, delta, mode, **kw)
            for key in ("row_ptr", "col", "val", "owner", "is_center", "lam_row"):
                assert np.array_equal(a[key], b[key]), (key, kw)


@pytest.mark.parametrize("gap", [1e-8, 1e-10, 1e-12])
@pytest.mark.parametrize("d,n,ell,m", [(2, 13, 2, 3), (2, 31, 4, 7), (3, 45, 3, 7)])
def test_nodes_nearer_than_rounding_are_no_error(gap, d, n, ell, m):
    """Such rows are lost to rounding in every solver; the others, whose stencils hold no pair, are
    the oracle's."""
    X = NS.disk2d(900, seed=3) if d == 2 else NS.ball3d(900, seed=3)
    rng = np.random.default_rng(3)
    v = rng.normal(size=(8, d))
    pairs = rng.choice(len(X), 8, replace=False)
    h = len(X) ** (-1.0 / d)
    Y = np.concatenate([X, X[pairs] + gap * h * v / np.linalg.norm(v, axis=1)[:, None]])
    g = gpu_run(Y, n, ell, m, 1.0)
    assert g["stats"]["n_singular"] == 0 and np.isfinite(g["val"]).all()
    ref = O.assemble(Y, n, ell, m, 1.0, R.STAB_SEQ)
    has = np.isin(ref["nbr"], np.arange(len(X), len(Y))).any(1)
    assert has.any() and not has.all()
    a, b = g["val"].reshape(-1, n), ref["val"].reshape(-1, n)
    err = np.linalg.norm(a - b, axis=1) / np.linalg.norm(b, axis=1)
    assert err[~has].max() < 1e-9
    # (a pair's weights cancel: of the size of its inverse gap at most)
    assert np.abs(a).max() <= 10.0 / gap * np.abs(b[~has]).max()


def test_nodes_on_a_line_stay_singular():
    X = np.stack([np.linspace(0.0, 1.0, 300), np.zeros(300)], 1)
    with R.Plan(torch.from_numpy(X).cuda(), 13, 2, 3, 1.0) as p:
        with pytest.raises(R.RbffdError) as e:
            p.assemble()
        assert e.value.code == R.ESINGULAR


@pytest.mark.parametrize("n,ell,m", [(27, 3, 7), (45, 3, 7), (30, 3, 7), (71, 4, 7), (113, 5, 7)])
def test_lattice_patches_in_other_node_sets(n, ell, m):
    """Too few lattice nodes for the plan to leave the null-space layout: their stencils alone are
    solved as saddle-point systems, at delta = 1 and with several columns."""
    side = 7
    X = np.concatenate([lattice(side, 3) + 10.0, NS.ball3d(6000, seed=6)])
    N, K = len(X), side ** 3
    g = gpu_run(X, n, ell, m, 1.0)
    assert g["stats"]["n_singular"] == 0
    ref = saddle(X, n, ell, m, 1.0)
    kind = np.array([constraints(X, g["nbr"][i], ell) for i in range(K)])
    assert (kind[:, 0] > 0).sum() > 0
    a = g["val"].reshape(N, n)[:-1]
    b = np.array([ref["val"][ref["row_ptr"][i]:ref["row_ptr"][i + 1]] for i in range(N - 1)])
    assert np.isfinite(a).all() and not np.array_equal(a, b)
    err = np.linalg.norm(a - b, axis=1) / np.linalg.norm(b, axis=1)
    assert err[:K][kind[:, 0] == 0].max(initial=0.0) < 1e-9 and err[K:].max() < 1e-9
    assert err[:K][(kind[:, 0] > 0) & (kind[:, 1] == 1)].max(initial=0.0) < 2e-8
    assert np.abs(a).max() <= 100.0 * np.abs(b).max()
    for mode in (R.STAB_OFF, R.STAB_FALLBACK):
        p = gpu_run(X, n, ell, m, 0.4, mode)
        assert p["stats"]["n_singular"] == 0 and np.isfinite(p["val"]).all()
        for kw in (dict(team=32, rhs_chunk=3), dict(team=256), dict(team=512, rhs_chunk=5)):
            q = gpu_run(X, n, ell, m, 0.4, mode, **kw)
            for key in ("val", "owner", "lam_row"):
                assert np.array_equal(p[key], q[key]), (key, kw)


def test_plans_of_lattices_have_the_saddle_point_layout():
    """The same bits as a plan of two shapes has, from a new plan and from one of another delta; turned
    and far from the origin too."""
    rot = np.linalg.qr(np.random.default_rng(1).normal(size=(3, 3)))[0]
    for X in (lattice(12, 3), lattice(12, 3) * np.array([1.0, 1.7, 2.3]) + 1000.0, lattice(12, 3) @ rot):
        t = torch.from_numpy(X).cuda()
        b = saddle(X, 45, 3, 7, 1.0)
        with R.Plan(t, 45, 3, 7, 0.5) as base, base.with_delta(1.0) as p:
            p.assemble()
            val = p.export()[2]
        assert np.array_equal(val[:45 * (len(X) - 1)], b["val"][:45 * (len(X) - 1)])
        assert np.array_equal(val, gpu_run(X, 45, 3, 7, 1.0)["val"])
