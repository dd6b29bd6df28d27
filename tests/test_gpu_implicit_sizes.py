"""Backward-Euler Newton on a thread-block cluster (block cyclic reduction) at sizes around its branches: one block
up to 11 elements, eight from 12 on; element counts at, below and above powers of two; one and two matrix columns per
lane (3 (2 (p + 1) + m3 + 1) + 1 columns); FP64 and FP32 factorization.

Tolerance 1e-11 relative L2 after two converged steps: the residual is FP64 in both, Newton stops at 1e-10 of the first
residual and its last iteration at least squares that, and rounding of these well-conditioned systems (dt = 1e-6) stays
near 1e-14.  Iteration counts may differ by one (the stopping test at the rounding floor); steps that do not converge
within the cap are those of the oracle.
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


@pytest.mark.parametrize("p,m3,mixed", [(1, 0, False), (1, 0, True), (2, 1, False), (2, 2, True), (3, 3, False)])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 11, 12, 16, 33, 64])
def test_sizes(n, p, m3, mixed):
    import paper_2301_11238_gb300 as G
    if mixed and 3 * (2 * (p + 1) + m3 + 1) > 30:
        pytest.skip("the FP32 factorization takes at most 10 unknowns a block")
    c = synth.paper_dam_break_1d(n_el=n, order=p, m3=m3)
    c.h_fn = lambda x, xc=None: 1.0 + 0.3 * np.sin(2.0 * x[:, 0])
    c.u_fn = lambda x, xc=None: 0.1 * np.cos(x)
    d, V0, _ = build(c)
    im = Implicit1D(d, 1e-6)
    Vh = d.to_modal(V0)
    X = im.pack(Vh, im.initial_E(Vh))
    s, _ = G.implicit_from_case(c, dt=1e-6, mixed=mixed)
    its = failed = 0
    for _ in range(2):
        X, it, ok = im.step(X)
        its += it
        failed += not ok
    st = s.run(2)
    V, E = s.get_state()
    Vo, _ = im.unpack(X)
    assert rel_l2(V, d.to_nodal(Vo)) < 1e-11
    assert abs(st["newton_its"] - its) <= 2 and st["failed_steps"] == failed
    assert np.isfinite(E).all()
