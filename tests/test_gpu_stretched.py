"""FP64 results on stretched triangles, component by component.

On elements of aspect ratio A the metric terms of the two directions differ by A, and
so do the gradient's and the residual's contributions; a computation may not let the
large ones take bits from the small ones.  The reference and the magnitude of each
result's sums are those of extended_residual.py.

Tolerance 64 units of 2^-53 times that magnitude: a dot product rounds once a term (at
most 10 + 12 of them at p = 3), metric terms are a few roundings old (10), and the
operator tables come from inverses in double precision (32).
"""
import numpy as np
import pytest

import extended_residual as X
import synth

pytestmark = pytest.mark.gpu

TOL = 64 * 2.0 ** -53
PRM = dict(g=9.81, rho=1.0, alpha=0.0, eta=0.05, sigma0=0.0, gamma=1.0, beta=1.0, pap_m=1.0, h_floor=1e-6, cfl=0.3,
           reg=0, positivity=0)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def mesh(aspect, along, shear):
    """5 x 5 squares in triangles, sheared, then stretched along one axis."""
    coords, etov = synth.rect_tri_mesh(5, 5)
    coords = coords.copy()
    coords[:, along] += shear * coords[:, 1 - along]
    coords[:, along] *= aspect
    return coords, etov


def both(coords, etov, p, V):
    """The library's and the reference's (dV/dt, E), the latter with magnitudes."""
    import paper_2301_11238_gb300 as G
    s = G.Solver(coords.shape[1], coords, etov, p, PRM["reg"], PRM)
    dV, E = s.residual(V)
    return dV.cpu().numpy(), E.cpu().numpy(), X.Rhs(coords, etov, p, PRM).rate(V)


def worst(x, ref, mag):
    """Largest error of each component in units of its magnitude."""
    return [float((np.abs(a - b) / np.where(m > 0, m, 1)).max()) for a, b, m in zip(x, ref, mag)]


def rough_state(K, p, seed=0):
    r = np.random.default_rng(seed).uniform(-1, 1, (3, K, (p + 1) * (p + 2) // 2))
    return np.stack([1 + 0.1 * r[0], 0.3 + 0.2 * r[1], -0.2 + 0.2 * r[2]])


@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("aspect", [1e3, 1e6])
@pytest.mark.parametrize("along", [0, 1])
@pytest.mark.parametrize("shear", [0.0, 0.5])
def test_gradient(p, aspect, along, shear):
    coords, etov = mesh(aspect, along, shear)
    V = rough_state(len(etov), p)
    _, E, (_, _, ref, mag) = both(coords, etov, p, V)
    assert max(worst(E, ref, mag)) < TOL


@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("aspect", [1.0, 1e3, 1e6])
@pytest.mark.parametrize("along", [0, 1])
@pytest.mark.parametrize("flow", ["fast", "slow", "one way"])
def test_residual(p, aspect, along, flow):
    """fast: velocities of the wave speed's size; slow: the pressure is nearly all there is; one way: one
    velocity component 1e-9 of the other."""
    coords, etov = mesh(aspect, along, 0.5)
    V = rough_state(len(etov), p)
    if flow == "slow":
        V[0] = 1.0
        V[1:] *= 1e-7
    if flow == "one way":
        V[2 - along] *= 1e-9
    dV, _, (ref, mag, _, _) = both(coords, etov, p, V)
    assert max(worst(dV, ref, mag)) < TOL


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("depth", [-1.0, -1e-3, 1e-9, "mixed"])
def test_depth_below_the_floor(dim, p, depth):
    """Elements whose depth is below the floor, alone and among wet ones: M_h then holds the floor, whatever
    the size of the nodal depths."""
    if dim == 1:
        coords, etov = np.linspace(0.0, 1.0, 41).reshape(-1, 1), np.stack([np.arange(40), np.arange(1, 41)], 1)
        etov = etov.astype(np.int32)
    else:
        coords, etov = mesh(1.0, 0, 0.0)
    r = np.random.default_rng(p).uniform(-1, 1, (3, len(etov), p + 1 if dim == 1 else (p + 1) * (p + 2) // 2))
    V = np.stack([1 + 0.1 * r[0], 0.3 + 0.2 * r[1], -0.2 + 0.2 * r[2]])[:dim + 1]
    if depth == "mixed":
        V[0, ::3] = 1e-9
        V[0, 1::3] *= -0.01
    else:
        V[0] *= depth
    dV, _, (ref, mag, _, _) = both(coords, etov, p, V)
    assert max(worst(dV, ref, mag)) < TOL
