"""Batch.set_state / get_state with device-side addresses: this GPU's memory (one launch) and any other memory that
CUDA can copy (field by field) give the same bytes; set_state can be captured."""
import ctypes as C

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def batch(precision, stream=None):
    import paper_2301_11238_gb300 as G
    return G.batch_from_cases([synth.radial_dam_2d(n=n, order=p) for n, p in ((3, 1), (7, 2), (5, 2), (4, 3))],
                              precision=precision, stream=stream)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("memory", ["device", "pinned"])
def test_round_trip(precision, memory):
    import torch
    b, V0s = batch(precision)
    rng = np.random.default_rng(0)
    for i, V0 in enumerate(V0s):
        V = rng.uniform(0.5, 1.0, V0.shape).astype(np.float32).astype(np.float64)
        x = torch.from_numpy(V)
        x = x.pin_memory() if memory == "pinned" else x.cuda()
        y = torch.empty_like(x, device="cuda") if memory == "device" else torch.empty(V.shape, dtype=torch.float64,
                                                                                      pin_memory=True)
        b._check(b.L.dg_batch_set_state(b.ctx, i, C.c_void_p(x.data_ptr()), 1))
        b._check(b.L.dg_batch_get_state(b.ctx, i, C.c_void_p(y.data_ptr()), 1))
        torch.cuda.synchronize()
        assert np.array_equal(y.cpu().numpy(), V) and np.array_equal(b.get_state(i), V)


@pytest.mark.parametrize("precision", [0, 1])
def test_set_state_in_a_capture(precision):
    import torch
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        b, V0s = batch(precision, s)
        x = [torch.from_numpy(V).cuda() for V in V0s]
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        g.capture_begin(capture_error_mode="global")
        for i, v in enumerate(x):
            b.set_state(i, v)
        g.capture_end()
        for v in x:
            v.mul_(0.5)
        g.replay()
        torch.cuda.synchronize()
        for i, V0 in enumerate(V0s):
            want = 0.5 * V0 if precision == 0 else (0.5 * V0).astype(np.float32)
            assert np.array_equal(b.get_state(i), want)
