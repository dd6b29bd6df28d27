"""Stable step and mass integral at element counts around the blocks of 256 and the partial sums, against numpy.

The step takes the wave speed at the node that a single-precision pass finds largest: it has to be the plain maximum's
value also for ties, for velocities outside the single-precision range and for states at rest.  Tolerances: FP64 step
8 roundings (square roots within 1 ulp, one quotient), FP32 step 1e-6 (8 roundings of 6e-8), mass 8 roundings of the
exact sum of the element integrals.
"""
import math

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def solver(K, p, precision, batch):
    import paper_2301_11238_gb300 as G
    c = synth.dam_break_1d(n_el=K, order=p, reg=0, sigma0=0.0, eta=0.0)
    if batch:
        return c, G.Batch([dict(dim=1, coords=c.coords, etov=c.etov, order=p, reg=0, prm=c.params, face_bc=c.face_bc,
                                bcs=c.bcs)] * 2, precision=precision)
    return c, G.Solver(1, c.coords, c.etov, p, 0, c.params, face_bc=c.face_bc, bcs=c.bcs, precision=precision)


def step_of(s, V, batch):
    if batch:
        s.set_state(0, V)
        s.set_state(1, V)
        st = s.run(1)
        assert st[0]["dt_last"] == st[1]["dt_last"]
        return st[0]
    s.set_state(V)
    return s.run(1)


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("K,p", [(1, 1), (31, 2), (33, 3), (255, 1), (256, 2), (257, 1), (1025, 3), (70001, 1)])
def test_step_and_mass(K, p, precision, batch):
    c, s = solver(K, p, precision, batch)
    rng = np.random.default_rng(K + p)
    g, cfl, q, dx = c.params["g"], c.params["cfl"], 2 * p + 1, np.diff(c.coords[:, 0])
    for kind in ("random", "ties", "rest", "extreme"):
        V = np.empty((2, K, p + 1))
        V[0] = 1.0 + rng.uniform(-0.5, 0.5, V[0].shape)
        V[1] = rng.uniform(-3, 3, V[1].shape)
        if kind == "ties":
            V[0], V[1] = 1.5, 0.25
        elif kind == "rest":
            V[1] = 0.0
        elif kind == "extreme":
            if precision:
                continue
            V[1] *= 10.0 ** rng.uniform(-60, 60, V[1].shape)
        lam = np.abs(V[1]) + np.sqrt(g * np.maximum(V[0], c.params["h_floor"]))
        want = (cfl * dx / (q * lam.max(axis=1))).min()
        w = {1: [1, 1], 2: [1 / 3, 4 / 3, 1 / 3], 3: [1 / 4, 3 / 4, 3 / 4, 1 / 4]}[p]
        st = step_of(s, V, batch) if kind != "extreme" else None
        if st is None:
            # the flow itself overflows in this step: only the step's size is looked at
            if batch:
                s.set_state(0, V)
                s.set_state(1, V)
                s.advance(1)
                st = s.stats()[0]
            else:
                s.set_state(V)
                st = dict(dt_last=s.step())
        else:
            R = np.float32 if precision else np.float64
            J = (0.5 * dx).astype(R).astype(float)
            m = math.fsum((J * (V[0].astype(R).astype(float) @ np.array(w))).tolist())
            assert abs(st["mass0"] - m) <= 8 * 1.2e-16 * m
        assert abs(st["dt_last"] - want) <= (1e-6 if precision else 8 * 1.2e-16) * want, kind


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_nonfinite_is_latched(precision, batch, bad):
    import paper_2301_11238_gb300 as G
    _, s = solver(300, 2, precision, batch)
    for field, e, a in ((0, 0, 0), (1, 299, 2), (1, 257, 1)):
        V = np.ones((2, 300, 3))
        V[field, e, a] = bad
        with pytest.raises(G.DGError) as err:
            step_of(s, V, batch)
        assert err.value.status == G.DG_ERR_NONFINITE
