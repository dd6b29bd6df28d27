"""dg_newton: what the workspace holds before a run, and on which stream it was set, does not matter; creating a
solver and giving it its workspace issue no CUDA work (a capture in the same thread stays whole)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def problem(stream=None):
    import paper_2301_11238_gb300 as G
    s, V0, _ = G.solver_from_case(synth.radial_dam_2d(n=8, order=2), stream=stream)
    return G, s, V0


def test_workspace_contents_do_not_matter():
    import torch
    G, s, V0 = problem()
    states = []
    for fill in (0, 255, 1):
        s.set_state(V0)
        nk = G.Newton(s, 1e-6)
        nk.workspace.fill_(fill)
        torch.cuda.synchronize()
        st = nk.run(2)
        states.append((s.get_state(with_E=False), st["krylov_its"], st["newton_its"]))
    for V, krylov, newton in states[1:]:
        assert np.array_equal(V, states[0][0]) and (krylov, newton) == states[0][1:]


@pytest.mark.parametrize("mode", ["thread_local", "global"])
def test_setup_leaves_a_capture_whole(mode):
    import torch
    own = torch.cuda.Stream()
    G, s, V0 = problem(own)
    x = torch.zeros(4, device="cuda")
    ws = torch.empty(1 << 24, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    p = G._lib.NewtonParams(dt=1e-6, max_newton=5, rtol=1e-8, atol=1e-10, krylov_dim=10, krylov_rtol=1e-3,
                            on_fail_continue=1)
    h = G.C.c_void_p()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(torch.cuda.Stream()):
        g.capture_begin(capture_error_mode=mode)
        y = x + 1
        status = [s.L.dg_newton_init(s.ctx, G.C.byref(p), G.C.byref(h))]
        assert s.L.dg_newton_workspace_size(h) <= ws.numel()
        status.append(s.L.dg_newton_set_workspace(h, G.C.c_void_p(ws.data_ptr()), ws.numel()))
        g.capture_end()
    s.L.dg_newton_destroy(h)
    assert status == [G.DG_OK, G.DG_OK]
    g.replay()
    torch.cuda.synchronize()
    assert bool((y == 1).all())
