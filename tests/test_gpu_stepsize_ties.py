"""The FP64 step bound's two steps (element_dt: single-precision speeds, then FP64 at the nodes near
their largest): speeds whose squares leave the single-precision range, and its time in still water.

Tolerance of the values as in test_gpu_stepsize.py (8 roundings).  Time: in still water of even depth
every node of an element is near the largest speed and is evaluated, 14 FP64 operations each for the 6
nodes of p = 2 beside about 25 of the element, in flow one or two of them: 109 operations against 39 to
53, so a limit of 2.5 to 2.8; FP32 evaluates every node in both (limit 1.25).
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("size", [1e-100, 1e-30, 3e-22, 1e-20, 1e-19, 1e-14, 1e-6, 1e17, 1e19, 1.9e19, 1e25, 1e100])
@pytest.mark.parametrize("p", [1, 3])
def test_speeds_of_any_size(p, size):
    import paper_2301_11238_gb300 as G
    K = 300
    c = synth.dam_break_1d(n_el=K, order=p, reg=0, sigma0=0.0, eta=0.0)
    c.params.update(h_floor=1e-300)
    s = G.Solver(1, c.coords, c.etov, p, 0, c.params, face_bc=c.face_bc, bcs=c.bcs)
    rng = np.random.default_rng(p)
    g, cfl, q, dx = c.params["g"], c.params["cfl"], 2 * p + 1, np.diff(c.coords[:, 0])
    V = np.empty((2, K, p + 1))
    # u and sqrt(g h) of the given size, and single nodes where one of them is nothing
    V[0] = (size * rng.uniform(0.9, 1.0, V[0].shape)) ** 2 / g
    V[1] = size * rng.uniform(0.9, 1.0, V[1].shape)
    V[0, :, 0] *= 1e-6
    V[1, ::2, 0] *= 1.01
    V[1, 1::3, -1] *= 1e-3
    lam = (np.abs(V[1]) + np.sqrt(g * V[0])).max(axis=1)
    s.set_state(V)
    dt = s.step()
    want = (cfl * dx / (q * lam)).min()
    assert abs(dt - want) <= 8 * 2.0 ** -52 * want, (dt, want)


@pytest.mark.parametrize("precision,limit", [(0, 2.8), (1, 1.25)])
def test_still_water_takes_no_longer(precision, limit):
    import paper_2301_11238_gb300 as G
    b, (V0,) = G.batch_from_cases([synth.slump_2d(n=512, order=2)], precision=precision)
    rng = np.random.default_rng(0)

    def dt_ms(rough):
        V = V0.copy()
        V[0] = 1.0 + rough * rng.uniform(-1, 1, V[0].shape)
        V[1:] = rough * rng.uniform(-1, 1, V[1:].shape)
        b.set_state(0, V)
        return min(b.time_kernels(30)[0]["dt"] for _ in range(5))

    flow, still = dt_ms(0.05), dt_ms(1e-15)
    assert still < limit * flow, (still, flow)
