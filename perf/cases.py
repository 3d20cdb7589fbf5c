"""The measured calls: what a user of the library has it do, from a 2,000-node disk to the
100,000-node ball, each through the public Python entry points.

Kinds of case:

* ``assemble``  -- stencils and differentiation matrices of a node set on the device, one matrix
  per overlap parameter (the first from ``Plan``, the others from ``Plan.with_delta``).
* ``mixed``     -- per-node stencil sizes and degrees in a clustered cube, FALLBACK stabilization,
  the matrix copied into buffers that hold the largest stencil in every row (how many entries it
  has is known after the call only).
* ``boundary``  -- Neumann boundary rows and the values of the time-stepping matrix.
* ``host``      -- nodes in host memory, matrix and stencil owners back in pinned host memory.
* ``apply``     -- y = L u with an assembled matrix, the step of an explicit time loop.
* ``stencils``  -- the allocation-free stencil step alone.

Degrees, stencil sizes and exponents are those of the node-set recipes and of the serving jobs:
n = 2 M + 1 nodes for M monomials (or the recipes' 12, 31 and 45), r^3 or r^5 with degree 2 and
r^7 above.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1606_03135_gb300 import nodesets as NS
from paper_1606_03135_gb300 import rbffd as R

BDF4_C = 12.0 / 25.0 * 1e-3  # (12/25) nu dt, nu = 1, dt = 1e-3


def terms(ell, d):
    return math.comb(ell + d, d)


def listed():
    return [
        # the smallest job: a 2D disk in one call, where launches and host time count
        dict(name="disk2d_small", kind="assemble", nodes="disk2d", N=2000, n=12, ell=2, m=3,
             deltas="0.5", mode=R.STAB_SEQ),
        # the 2D workload: three overlap parameters of one node set
        dict(name="square2d_sweep", kind="assemble", nodes="square2d", N=40000, n=31, ell=4, m=7,
             deltas="1.0 0.5 0.3", mode=R.STAB_SEQ),
        # the 3D workload of the benchmark
        dict(name="ball3d_sweep", kind="assemble", nodes="ball3d", N=100000, n=45, ell=3, m=7,
             deltas="1.0 0.4 0.2", mode=R.STAB_SEQ),
        # standard RBF-FD (one stencil per node) of a small 3D set of ragged size
        dict(name="ball3d_standard", kind="assemble", nodes="ball3d", N=5003, n=45, ell=3, m=7,
             deltas="1.0", mode=R.STAB_SEQ),
        # higher degrees in 3D, as the serving jobs ask for them
        dict(name="ball3d_degree4", kind="assemble", nodes="ball3d", N=12000, n=71, ell=4, m=7,
             deltas="0.4", mode=R.STAB_SEQ),
        dict(name="ball3d_degree5", kind="assemble", nodes="ball3d", N=4001, n=113, ell=5, m=7,
             deltas="0.6", mode=R.STAB_SEQ),
        # per-node degrees 2..5 with FALLBACK re-solves
        dict(name="cube3d_mixed", kind="mixed", nodes="cube3d", N=20000, deltas="0.3"),
        # Neumann disk: interior and boundary rows, then I - c L
        dict(name="disk2d_neumann", kind="boundary", nodes="disk2d_bc", N=10000, n=31, ell=4, m=7,
             deltas="0.5", mode=R.STAB_SEQ),
        # a serving job: host nodes in, host matrix out
        dict(name="disk2d_host_job", kind="host", nodes="disk2d", N=30011, n=43, ell=5, m=7,
             deltas="0.6", mode=R.STAB_SEQ),
        # y = L u of the 3D workload and of the small disk
        dict(name="apply_ball3d", kind="apply", nodes="ball3d", N=100000, n=45, ell=3, m=7,
             deltas="1.0", mode=R.STAB_SEQ),
        dict(name="apply_disk2d_small", kind="apply", nodes="disk2d", N=2000, n=12, ell=2, m=3,
             deltas="0.5", mode=R.STAB_SEQ),
        # stencils only, into the caller's buffers
        dict(name="stencils_ball3d", kind="stencils", nodes="ball3d", N=20000, n=45, deltas="0.4"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["assemble"] * 5 + ["mixed", "boundary", "host", "apply", "stencils"])
    if kind == "mixed":
        return dict(kind=kind, nodes="cube3d", N=log_int(3000, 20000),
                    deltas="%.3f" % rng.uniform(0.25, 0.6))
    if kind == "stencils":
        d = rng.choice([2, 3])
        ell = rng.randint(2, 5)
        n = 2 * terms(ell, d) + 1
        return dict(kind=kind, nodes="disk2d" if d == 2 else "ball3d", N=log_int(max(1000, n), 32768),
                    n=n, deltas="%.3f" % rng.uniform(0.2, 1.0))
    d = 2 if kind == "boundary" else rng.choice([2, 3])
    ell = rng.randint(2, 5)
    n = 2 * terms(ell, d) + 1
    if kind != "apply" and rng.random() < 0.3:  # a stencil size of the user's own choice
        n = rng.randint(terms(ell, d) + terms(ell, d) // 2, min(128, n + 8))
    m = rng.choice([3, 5]) if ell == 2 else 7
    # no dearer than the 3D workload: bounded by the factorizations of one stencil per node
    top = int(3e10 / (n + terms(ell, d)) ** 3)
    N = log_int(1000, max(1500, min(100000, top)))
    deltas = ["%.3f" % rng.uniform(0.2, 1.0)]
    if kind == "assemble" and rng.random() < 0.3:
        deltas = ["1.0"] + deltas
    nodes = "disk2d_bc" if kind == "boundary" else "disk2d" if d == 2 else "ball3d"
    return dict(kind=kind, nodes=nodes, N=N, n=n, ell=ell, m=m, deltas=" ".join(deltas),
                mode=rng.choice([R.STAB_SEQ, R.STAB_SEQ, R.STAB_FALLBACK])
                if kind == "assemble" else R.STAB_SEQ)


def _nodes(case, seed):
    """(X, bc, normals) of a case on the host."""
    gen, N = case["nodes"], case["N"]
    if gen == "disk2d_bc":
        return NS.disk2d_bc(N, seed=seed)
    X = {"disk2d": NS.disk2d, "ball3d": NS.ball3d, "square2d": NS.square2d,
         "cube3d": NS.cube3d_clustered}[gen](N, seed=seed)
    return X, None, None


def _deltas(case):
    return [float(t) for t in case["deltas"].split()]


def prepare(case, seed):
    kind = case["kind"]
    X, bc, normals = _nodes(case, seed)
    st = dict(case=case, deltas=_deltas(case))
    N = X.shape[0]
    if kind == "host":
        st["X"] = X
        n = case["n"]
        pin = lambda size, dt: torch.empty(size, dtype=dt, pin_memory=True).numpy()
        st["out"] = (pin(N + 1, torch.int64), pin(N * n, torch.int32), pin(N * n, torch.float64),
                     pin(N, torch.int32))
        return st
    st["X"] = torch.from_numpy(X).cuda()
    if kind == "mixed":
        st["params"] = NS.mixed_degree_params(X)
        st["col"] = torch.zeros(N * 113, dtype=torch.int32, device="cuda")
        st["val"] = torch.zeros(N * 113, dtype=torch.float64, device="cuda")
    elif kind == "boundary":
        st["bc"], st["normals"] = bc, normals
    elif kind == "apply":
        st["plan"] = R.Plan(st["X"], case["n"], case["ell"], case["m"], st["deltas"][0],
                            mode=case["mode"])
        st["plan"].assemble()
        st["u"] = torch.from_numpy(_field(X)).cuda()
        st["y"] = torch.empty(N, dtype=torch.float64, device="cuda")
    elif kind == "stencils":
        st["nbr"] = torch.empty(N, case["n"], dtype=torch.int32, device="cuda")
        st["rho2"] = torch.empty(N, dtype=torch.float64, device="cuda")
        st["ball"] = torch.empty(N, dtype=torch.int32, device="cuda")
    return st


def _field(X):
    """A smooth field at the nodes (the u of y = L u)."""
    return np.sin(3.0 * X[:, 0] + 0.5) * np.cos(2.0 * X[:, 1]) + (X[:, -1] - 0.25) ** 3


class _View:
    """A device array of the library as torch.as_tensor takes it (no copy).  The tensor keeps
    this object, and with it the plan that owns the memory."""

    def __init__(self, plan, ptr, size, typestr):
        self.plan = plan
        self.__cuda_array_interface__ = dict(shape=(size,), typestr=typestr, data=(ptr, False),
                                             version=3)


def _matrix_of(plan):
    """Assemble, and the matrix as device tensors."""
    csr = plan.assemble()
    view = lambda ptr, size, t: torch.as_tensor(_View(plan, ptr, size, t), device="cuda")
    return dict(row_ptr=view(csr.row_ptr, csr.n_rows + 1, "<i8"), col=view(csr.col, csr.nnz, "<i4"),
                val=view(csr.val, csr.nnz, "<f8"))


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "apply":
        st["plan"].apply(st["u"], st["y"])
        return st["y"]
    if kind == "stencils":
        X = st["X"]
        rc = R.rbffd_stencils_noalloc(X, X.shape[0], X.shape[1], case["n"], st["deltas"][0],
                                      st["nbr"], st["rho2"], st["ball"],
                                      torch.cuda.current_stream().cuda_stream)
        if rc != R.OK:
            raise R.RbffdError(rc, "rbffd_stencils_noalloc")
        return dict(nbr=st["nbr"], rho2=st["rho2"], ball=st["ball"])
    if kind == "host":
        with R.Plan(st["X"], case["n"], case["ell"], case["m"], st["deltas"][0],
                    mode=case["mode"]) as p:
            p.assemble()
            row_ptr, col, val, owner = p.export(st["out"])
        return dict(row_ptr=row_ptr, col=col, val=val, owner=owner)
    if kind == "mixed":
        p = R.Plan(st["X"], *st["params"], st["deltas"][0], mode=R.STAB_FALLBACK)
        out = _matrix_of(p)
        for name in ("col", "val"):
            st[name][:out[name].numel()] = out[name]
            out[name] = st[name]
        return out
    if kind == "boundary":
        p = R.Plan(st["X"], case["n"], case["ell"], case["m"], st["deltas"][0], mode=case["mode"])
        p.set_boundary(st["bc"], st["normals"])
        out = _matrix_of(p)
        out["step"] = p.timestep_matrix(BDF4_C)
        return out
    first, outs = None, []
    for delta in st["deltas"]:
        if first is None:
            p = first = R.Plan(st["X"], case["n"], case["ell"], case["m"], delta, mode=case["mode"])
        else:
            p = first.with_delta(delta, mode=case["mode"])
        outs.append(_matrix_of(p))
    return outs


def _rows(case):
    """(rows, dimension) of a case's matrix; boundary sets carry two rings of 2 pi / h nodes."""
    d = 3 if case["nodes"] in ("ball3d", "cube3d") else 2
    N = case["N"]
    if case["nodes"] == "disk2d_bc":
        N += 2 * int(round(2.0 * math.pi / math.sqrt(math.pi / N)))
    return N, d


def work(case):
    """Bytes: nodes in, matrices out (and its vectors for y = L u).  Flops: one symmetric
    factorization per stencil, K^3 / 3, with at most the ball's (1 - delta)^d n rows from each,
    and one solve, 2 K^2, per row."""
    N, d = _rows(case)
    kind = case["kind"]
    if kind == "mixed":  # four slabs of degree 2..5, a quarter of the nodes each
        M = [terms(l, d) for l in (2, 3, 4, 5)]
        shapes = [(N / 4, 2 * k + 1, 3 * k + 1) for k in M]
    else:
        n = case["n"]
        shapes = [(N, n, n + (terms(case["ell"], d) if "ell" in case else 0))]
    nnz = sum(c * n for c, n, _ in shapes)
    if kind == "apply":
        return dict(bytes=nnz * 12 + N * 24, flops=2 * nnz)
    if kind == "stencils":
        return dict(bytes=N * d * 8 + nnz * 4 + N * 12, flops=nnz * (3 * d - 1))
    b = f = 0.0
    for delta in _deltas(case):
        b += N * d * 8 + nnz * 12 + N * 8 + (nnz * 8 if kind == "boundary" else 0)
        for c, n, K in shapes:
            f += c / max((1.0 - delta) ** d * n, 1.0) * K ** 3 / 3.0 + c * 2.0 * K * K
    return dict(bytes=b, flops=f)


# ------------------------------------------------------------------ the results in plain numpy
def _knn(X, n):
    """(N, n) neighbours by (squared distance, index) and their squared distances."""
    N = X.shape[0]
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    T = torch.from_numpy(X).to(dev)
    nbr, d2 = np.empty((N, n), np.int64), np.empty((N, n))
    for i0 in range(0, N, 2048):
        D = torch.zeros(min(2048, N - i0), N, dtype=torch.float64, device=dev)
        for a in range(X.shape[1]):
            t = T[i0:i0 + 2048, a, None] - T[None, :, a]
            D += t * t
        v, idx = torch.topk(D, min(N, n + 8), dim=1, largest=False)
        v, idx = v.cpu().numpy(), idx.cpu().numpy()
        o = np.lexsort((idx, v), axis=1)[:, :n]
        nbr[i0:i0 + 2048] = np.take_along_axis(idx, o, 1)
        d2[i0:i0 + 2048] = np.take_along_axis(v, o, 1)
    return nbr, d2


def _exponents(ell, d):
    return np.array([e for e in np.ndindex(*([ell + 1] * d)) if sum(e) <= ell])


def _systems(x, m, E):
    """Saddle-point matrices of stencils x (B, n, d) in scaled coordinates."""
    B, n, d = x.shape
    r2 = ((x[:, :, None] - x[:, None]) ** 2).sum(-1)
    M = len(E)
    S = np.zeros((B, n + M, n + M))
    S[:, :n, :n] = r2 ** 3 * np.sqrt(r2) if m == 7 else np.sqrt(r2) ** m
    P = np.prod(x[:, :, None] ** E[None, None], axis=-1)
    S[:, :n, n:] = P
    S[:, n:, :n] = P.transpose(0, 2, 1)
    return S


def _laplacian(x, y, m, E):
    """Right-hand sides (B, n + M, q): the Laplacian of every basis function at y (B, q, d)."""
    B, n, d = x.shape
    r = np.sqrt(((x[:, :, None] - y[:, None]) ** 2).sum(-1))
    low = np.zeros((B, len(E), y.shape[1]))
    for a in range(d):
        D = E.copy()
        D[:, a] -= 2
        ok = D[:, a] >= 0
        c = (E[ok, a] * (E[ok, a] - 1)).astype(np.float64)
        low[:, ok] += c[:, None] * np.prod(y[:, None] ** D[ok][None, :, None], axis=-1)
    return np.concatenate([m * (m + d - 2) * r ** (m - 2), low], axis=1)


def _matrix(X, n, ell, m, delta, mode, bc=None, normals=None):
    """Values of L with ascending columns in every row, rows one after the other (n, ell, m per
    node), from numpy's LU of every local system."""
    N, d = X.shape
    nmax = int(n.max())
    nbr, d2 = _knn(X, nmax)
    rho2 = d2[np.arange(N), n - 1]
    rho = np.sqrt(rho2)
    ball = [int((d2[k, :n[k]] <= (1.0 - delta) * (1.0 - delta) * rho2[k]).sum()) for k in range(N)]
    tables = {int(l): _exponents(int(l), d) for l in set(ell.tolist())}
    rows = [None] * N
    bc = np.zeros(N, np.uint8) if bc is None else bc

    def solve(ks, members):
        """Weights (len(ks), n, q) at the member positions of stencils ks of one shape."""
        k0 = ks[0]
        E = tables[int(ell[k0])]
        idx = nbr[ks, :n[k0]]
        x = (X[idx] - X[ks][:, None]) / rho[ks][:, None, None]
        y = np.take_along_axis(x, members[:, :, None], 1)
        w = np.linalg.solve(_systems(x, int(m[k0]), E), _laplacian(x, y, int(m[k0]), E))
        return w[:, :n[k0]]

    def own(ks):
        """Own-stencil rows, in batches of one shape."""
        for s in sorted({(int(n[k]), int(ell[k]), int(m[k])) for k in ks}):
            kk = np.array([k for k in ks if (n[k], ell[k], m[k]) == s])
            for b in range(0, len(kk), 1024):
                part = kk[b:b + 1024]
                w = solve(part, np.zeros((len(part), 1), np.int64))
                for k, v in zip(part, w[:, :, 0]):
                    rows[k] = (k, v / rho2[k])

    for k in np.flatnonzero(bc):  # Dirichlet and Neumann rows from their own stencils
        k = int(k)
        e = np.zeros(n[k])
        e[0] = 1.0
        if bc[k] == 2:
            E = tables[int(ell[k])]
            x = ((X[nbr[k, :n[k]]] - X[k]) / rho[k])[None]
            r = np.sqrt((x ** 2).sum(-1))[0]
            f = np.zeros(n[k] + len(E))
            f[:n[k]] = -m[k] * r ** (int(m[k]) - 2) * (x[0] @ normals[k])
            for a in range(d):
                f[n[k] + int(np.flatnonzero((E.sum(1) == 1) & (E[:, a] == 1))[0])] = normals[k, a]
            e = np.linalg.solve(_systems(x, int(m[k]), E)[0], f)[:n[k]] / rho[k]
        rows[k] = (k, e)
    if delta >= 1.0:
        own([k for k in range(N) if rows[k] is None])
    else:
        redo = []
        for k in range(N):
            if rows[k] is not None:
                continue
            mem = np.array([t for t in range(ball[k])
                            if t == 0 or (nbr[k, t] > k and rows[nbr[k, t]] is None)])
            w = solve(np.array([k]), mem[None])[0]
            lam = np.abs(w).sum(0)
            for c, t in enumerate(mem):
                if c == 0 or mode != R.STAB_SEQ or lam[c] <= lam[0]:
                    rows[nbr[k, t]] = (k, w[:, c] / rho2[k])
                if c and mode == R.STAB_FALLBACK and lam[c] > lam[0]:
                    redo.append(int(nbr[k, t]))
        own(redo)
    out = []
    for k, v in rows:
        out.append(v[np.argsort(nbr[k, :len(v)])])
    return np.concatenate(out), rows, nbr


def exact(case, seed):
    kind = case["kind"]
    X, bc, normals = _nodes(case, seed)
    N = X.shape[0]
    deltas = _deltas(case)
    if kind == "stencils":
        nbr, d2 = _knn(X, case["n"])
        return dict(nbr=None, rho2=d2[:, -1], ball=None)
    if kind == "mixed":
        n, ell, m = NS.mixed_degree_params(X)
    else:
        n, ell, m = (np.full(N, case[s], np.int64) for s in ("n", "ell", "m"))
    K = int(n.max()) + terms(int(ell.max()), X.shape[1])
    cost = [N * (2e-5 + (K / 65.0) ** 3 * (6e-5 if delta >= 1.0 else 2.5e-4)) for delta in deltas]
    mode = R.STAB_FALLBACK if kind == "mixed" else case["mode"]
    vals, spent = [], 0.0
    for delta, c in zip(deltas, cost):
        spent += c
        vals.append(_matrix(X, n, ell, m, delta, mode, bc, normals) if spent < 18.0 else None)
    if all(v is None for v in vals):
        return None
    if kind == "assemble":
        return [v if v is None else dict(row_ptr=None, col=None, val=v[0]) for v in vals]
    val, rows, nbr = vals[0]
    if kind == "apply":
        u = _field(X)
        return np.array([v @ u[nbr[k, :len(v)]] for k, v in rows])
    if kind == "mixed":
        val = np.concatenate([val, np.zeros(N * 113 - val.size)])
    out = dict(row_ptr=None, col=None, val=val)
    if kind == "host":
        out["owner"] = None
    if kind == "boundary":
        step = []
        for i, (k, v) in enumerate(rows):
            c = np.sort(nbr[k, :len(v)])
            w = v[np.argsort(nbr[k, :len(v)])]
            step.append(w if bc[i] else (c == i) - BDF4_C * w)
        out["step"] = np.concatenate(step)
    return out
