"""Block fixed-point contractions of the FP64 kernels (csrc/dg_fixed.cuh) away from
smooth states of size 1: rough fields of very large and very small size,
single nodes far above the rest, exact zeros, and non-finite values.

The reference for E is exact: the strong nodal form E = grad u + LIFT(n [u]/2)
in rational arithmetic on the same doubles.  (The oracle's modal basis spreads
the rounding of a large nodal value over its element.)  Tolerance 1e-13
relative L2: a result is a sum of at most a few dozen terms of its own size,
with metric terms rounded to doubles (1.1e-16 each); the fixed-point side drops
less than 2^-55 of the largest term per sum.
"""
from fractions import Fraction as Q

import numpy as np
import pytest

from helpers import both, rel_l2, smooth_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def rough_case(dim, p, bc="copy"):
    c = smooth_case(dim, p, 0, n=40 if dim == 1 else 5, seed=p, bc=bc)
    return (c,) + both(c)


def solve(A, B):
    """X of A X = B over the rationals (Gauss-Jordan; A square, B a matrix)."""
    n = len(A)
    M = [list(A[i]) + list(B[i]) for i in range(n)]
    for k in range(n):
        i = next(i for i in range(k, n) if M[i][k] != 0)
        M[k], M[i] = M[i], M[k]
        M[k] = [x / M[k][k] for x in M[k]]
        for i in range(n):
            if i != k and M[i][k] != 0:
                M[i] = [x - M[i][k] * y for x, y in zip(M[i], M[k])]
    return [row[n:] for row in M]


def reference_operators(dim, p):
    """Derivative matrices and LIFT per face (rows of node, columns of the face's nodes), exact."""
    ex = [(i, 0) for i in range(p + 1)] if dim == 1 else [(i, j) for j in range(p + 1) for i in range(p + 1 - j)]
    node = [(Q(2 * i, p) - 1, Q(2 * j, p) - 1 if dim == 2 else Q(0)) for i, j in ex]
    n = len(node)
    mono = [[r ** a * s ** b for a, b in ex] for r, s in node]
    C = solve(mono, [[Q(int(i == j)) for j in range(n)] for i in range(n)])  # column a: coefficients of l_a

    def integral(a, b):  # of r^a s^b over the reference element
        if dim == 1:
            return Q(1 - (-1) ** (a + 1), a + 1)
        # r from -1 to -s: int s^b ((-s)^(a+1) - (-1)^(a+1)) / (a+1) ds over [-1, 1]
        one = lambda k: Q(1 - (-1) ** (k + 1), k + 1)  # noqa: E731
        return Q((-1) ** (a + 1), a + 1) * (one(a + b + 1) - one(b))

    def product(i, j, der=None):  # <l_i, l_j>, or <l_i, d l_j / d der>
        t = Q(0)
        for k, (a, b) in enumerate(ex):
            for m, (c, d) in enumerate(ex):
                if der is None:
                    t += C[k][i] * C[m][j] * integral(a + c, b + d)
                elif der == 0 and c:
                    t += c * C[k][i] * C[m][j] * integral(a + c - 1, b + d)
                elif der == 1 and d:
                    t += d * C[k][i] * C[m][j] * integral(a + c, b + d - 1)
        return t

    M = [[product(i, j) for j in range(n)] for i in range(n)]
    D = [solve(M, [[product(i, j, der) for j in range(n)] for i in range(n)]) for der in range(dim)]
    if dim == 1:
        faces = [[0], [p]]
        edge = [[Q(1)]]
    else:
        at = {x: a for a, x in enumerate(ex)}
        faces = [[at[k, 0] for k in range(p + 1)], [at[p - k, k] for k in range(p + 1)],
                 [at[0, p - k] for k in range(p + 1)]]
        t = [Q(2 * k, p) - 1 for k in range(p + 1)]
        E = solve([[x ** k for k in range(p + 1)] for x in t],
                  [[Q(int(i == j)) for j in range(p + 1)] for i in range(p + 1)])
        edge = [[sum(E[k][i] * E[m][j] * Q(1 - (-1) ** (k + m + 1), k + m + 1) for k in range(p + 1)
                     for m in range(p + 1)) for j in range(p + 1)] for i in range(p + 1)]
    lift = []
    for f in faces:
        rows = [[Q(0)] * len(f) for _ in range(n)]
        for i, a in enumerate(f):
            rows[a] = edge[i]
        lift.append(solve(M, rows))
    return D, lift, faces


def exact_gradient(c, V, wall):
    """E (dim^2, K, Np) of the nodal state V on case c; copy or wall boundaries."""
    dim, K, Np = c.dim, V.shape[1], V.shape[2]
    D, lift, faces = reference_operators(dim, c.order)
    u = [[[Q(float(x)) for x in row] for row in V[1 + j]] for j in range(dim)]
    X = [[Q(float(x)) for x in row] for row in c.coords]
    where = {}
    for e, ev in enumerate(c.etov):
        for f in range(dim + 1):
            key = (int(ev[f]),) if dim == 1 else tuple(sorted((int(ev[f]), int(ev[(f + 1) % 3]))))
            where.setdefault(key, []).append((e, f))
    other = {}
    for pair in where.values():
        if len(pair) == 2:
            other[pair[0]], other[pair[1]] = pair[1], pair[0]
    E = np.zeros((dim * dim, K, Np))
    for e, ev in enumerate(c.etov):
        v = [X[i] for i in ev]
        if dim == 1:
            J = (v[1][0] - v[0][0]) / 2
            G, area = [[1 / J]], [[Q(-1)], [Q(1)]]  # area: normal times face Jacobian
        else:
            xr, yr, xs, ys = ((v[k][d] - v[0][d]) / 2 for k in (1, 2) for d in (0, 1))
            J = xr * ys - xs * yr
            G = [[ys / J, -xs / J], [-yr / J, xr / J]]
            area = [[(v[(f + 1) % 3][1] - v[f][1]) / 2, (v[f][0] - v[(f + 1) % 3][0]) / 2] for f in range(3)]
        out = [[[Q(0)] * Np for _ in range(dim)] for _ in range(dim)]
        for j in range(dim):
            for r in range(dim):
                for a in range(Np):
                    d = sum(D[r][a][b] * u[j][e][b] for b in range(Np))
                    for i in range(dim):
                        out[i][j][a] += G[r][i] * d
        for f in range(dim + 1):
            own = faces[f]
            if (e, f) in other:
                e2, f2 = other[e, f]
                ext = [[u[j][e2][b] for b in reversed(faces[f2])] for j in range(dim)]
            else:
                ext = [[u[j][e][a] for a in own] for j in range(dim)]
                if wall:
                    nn = sum(x * x for x in area[f])
                    for k in range(len(own)):
                        un = sum(ext[j][k] * area[f][j] for j in range(dim))
                        for j in range(dim):
                            ext[j][k] -= 2 * un * area[f][j] / nn
            for j in range(dim):
                jump = [(x - u[j][e][a]) / 2 for x, a in zip(ext[j], own)]
                for a in range(Np):
                    w = sum(L * g for L, g in zip(lift[f][a], jump))
                    for i in range(dim):
                        out[i][j][a] += area[f][i] / J * w
        for i in range(dim):
            for j in range(dim):
                E[dim * i + j, e] = [float(x) for x in out[i][j]]
    return E


@pytest.mark.parametrize("dim,p", [(1, 1), (1, 3), (2, 1), (2, 2), (2, 3)])
def test_exact_gradient_is_the_oracles(dim, p):
    from oracle.run import residual_nodal
    c, d, V0, _, _ = rough_case(dim, p, "wall")
    assert rel_l2(exact_gradient(c, V0, True), residual_nodal(d, V0)[1]) < 1e-12


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("bc", ["copy", "wall"])
def test_gradient_of_rough_velocities(dim, p, bc):
    c, _, V0, _, s = rough_case(dim, p, bc)
    rng = np.random.default_rng(10 * p + dim)
    for scale in (1.0, 1e-200, 1e-20, 1e20, 1e140):
        V = V0.copy()
        V[1:] = scale * rng.uniform(-1, 1, V[1:].shape)
        V[1:][:, ::7] = 0.0                # elements exactly at rest
        V[1:, 3, 0] *= 1e9                 # one node far above its element
        V[1:, 11, -1] *= 1e-30             # and one far below
        E_o = exact_gradient(c, V, bc == "wall")
        _, E = s.residual(V)
        E = E.cpu().numpy()
        # the spiked element and its neighbours separately, so that they do not hide the rest
        big = np.abs(E_o).max(axis=(0, 2)) > 1e4 * np.median(np.abs(E_o).max(axis=(0, 2)))
        for part in (big, ~big):
            assert rel_l2(E[:, part], E_o[:, part]) < 1e-13, (scale, part.sum())


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_rest_is_exact(dim, p):
    _, _, V0, _, s = rough_case(dim, p)
    V = V0.copy()
    V[1:] = 0.0
    _, E = s.residual(V)
    assert float(E.abs().max()) == 0.0


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_nonfinite_stays_nonfinite(dim, p, bad):
    _, _, V0, _, s = rough_case(dim, p)
    for field in range(dim + 1):
        V = V0.copy()
        V[field, 9, 0] = bad
        dV, E = s.residual(V)
        dV, E = dV.cpu().numpy(), E.cpu().numpy()
        assert not np.isfinite(dV[field, 9]).any()
        if field > 0:
            assert not np.isfinite(E[:, 9]).all()
        far = np.ones(V.shape[1], dtype=bool)
        far[max(0, 9 - 25):9 + 25] = False
        assert np.isfinite(dV[:, far]).all() and np.isfinite(E[:, far]).all()
