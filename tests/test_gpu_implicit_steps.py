"""The 1D Newton integrator's block cyclic reduction where the off-diagonal blocks matter: steps of ten explicit bounds
and more, at element counts around the cluster's line and powers of two, every block size.

Tolerance 1e-9 relative L2 after two steps: both stop once the residual has fallen by 1e-10, and the last iteration
of Newton at least squares that; elimination orders differ, and their rounding is that of the condition of the
Jacobian, below 1e6 here, times 2^-53.
"""
import numpy as np
import pytest

import synth
from helpers import rel_l2
from oracle.implicit import Implicit1D
from oracle.run import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("p,m3,mixed", [(1, 0, False), (1, 1, True), (2, 1, False), (2, 2, True), (3, 3, False)])
@pytest.mark.parametrize("n", [2, 7, 11, 12, 31, 32, 33, 100])
def test_large_steps(n, p, m3, mixed):
    import paper_2301_11238_gb300 as G
    c = synth.paper_dam_break_1d(n_el=n, order=p, m3=m3, gamma=5.0, beta=20.0)
    c.h_fn = lambda x, xc=None: 1.0 + 0.2 * np.sin(2.0 * x[:, 0])
    c.u_fn = lambda x, xc=None: 0.3 * np.cos(x)
    d, V0, _ = build(c)
    Vh = d.to_modal(V0)
    dt = 10.0 * d.stable_dt(Vh)
    im = Implicit1D(d, dt)
    X = im.pack(Vh, im.initial_E(Vh))
    its = failed = 0
    for _ in range(2):
        X, it, ok = im.step(X)
        its += it
        failed += not ok
    s, _ = G.implicit_from_case(c, dt=dt, mixed=mixed)
    st = s.run(2)
    V, _ = s.get_state()
    Vo = d.to_nodal(im.unpack(X)[0])
    assert rel_l2(Vo, V0) > 1e-4  # the steps do something
    if failed == 0:
        assert rel_l2(V, Vo) < 1e-9
        assert st["failed_steps"] == 0 and abs(st["newton_its"] - its) <= 2
    else:
        assert st["failed_steps"] == failed
