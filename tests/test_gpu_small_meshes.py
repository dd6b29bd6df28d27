"""FP64 paths chosen by mesh size: the volume pass with several lanes per element (up to 152 x 4 x 32 = 19,456
elements) against the one with a thread per element, and the lane groups of the Newton-Krylov kernels.

Both volume forms add the same integers, so results agree bit for bit: a small instance alone (lanes) and the same
instance in a batch whose group is beyond the line (a thread per element).
"""
import numpy as np
import pytest

import synth
from helpers import rel_l2, smooth_case
from oracle.implicit_reduced import ImplicitReduced
from oracle.run import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def spec(c, bed):
    return dict(dim=c.dim, coords=c.coords, etov=c.etov, order=c.order, reg=c.params["reg"], prm=c.params,
                face_bc=c.face_bc, bcs=c.bcs, bed=bed if c.bed_fn is not None else None)


@pytest.mark.parametrize("dim,p", [(1, 1), (1, 2), (1, 3), (2, 1), (2, 2), (2, 3)])
@pytest.mark.parametrize("n,bed", [(1, False), (3, True), (7, True), (31, False)])
def test_lanes_equal_thread_per_element(dim, p, n, bed):
    import paper_2301_11238_gb300 as G
    c = smooth_case(dim, p, 3, n=n if dim == 2 else n + 1, seed=p, bed=bed, bc="wall")
    d, V0, b = build(c)
    big = synth.dam_break_1d(n_el=19500, order=p) if dim == 1 else synth.radial_dam_2d(n=99, order=p)
    _, Vb, _ = build(big)
    alone = G.Batch([spec(c, b)])
    alone.set_state(0, V0)
    group = G.Batch([spec(c, b), spec(big, None)])
    group.set_state(0, V0)
    group.set_state(1, Vb)
    alone.run(3)
    group.run(3)
    assert np.array_equal(alone.get_state(0), group.get_state(0))


@pytest.mark.parametrize("dim,p", [(1, 1), (1, 3), (2, 1), (2, 3)])
@pytest.mark.parametrize("n", [1, 2, 5])
def test_newton_krylov_sizes(dim, p, n):
    """One step against the reduced oracle, 1e-9 (the Newton stopping rule, as in the solver's other tests)."""
    import paper_2301_11238_gb300 as G
    c = smooth_case(dim, p, 3, n=n if dim == 2 else 3 * n, seed=3, gamma=5.0, bed=False)
    d, V0, _ = build(c)
    dt = 5.0 * d.stable_dt(d.to_modal(V0))
    V1, _, _ = ImplicitReduced(d, dt).step(d.to_modal(V0), rtol=1e-14, atol=1e-11)
    s, _, _ = G.solver_from_case(c)
    G.Newton(s, dt, rtol=1e-13, atol=1e-11, krylov_dim=64, krylov_rtol=1e-11).run(1)
    assert rel_l2(s.get_state(with_E=False), d.to_nodal(V1)) < 1e-9
