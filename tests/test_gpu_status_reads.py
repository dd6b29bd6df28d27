"""Status reads (dg_swe_sync, dg_swe_get_state, dg_batch_stats) by several threads of one context at a time."""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_concurrent_reads_of_one_context():
    import torch
    import paper_2301_11238_gb300 as G
    s, V0, _ = G.solver_from_case(synth.radial_dam_2d(n=16, order=2))
    b, Vs = G.batch_from_cases([synth.radial_dam_2d(n=16, order=2)] * 3)
    s.run(3)
    b.run(3)
    want, want_b, V = s.sync(), b.stats(), s.get_state(with_E=False)
    bad = []

    def read(k):
        out = torch.empty(V0.shape, dtype=torch.float64, device="cuda")
        for _ in range(50):
            if s.sync() != want or b.stats() != want_b:
                bad.append(k)
            s.get_state_device(out)
            if not np.array_equal(out.cpu().numpy(), V):
                bad.append(k)

    t = [threading.Thread(target=read, args=(k,)) for k in range(6)]
    [x.start() for x in t]
    [x.join() for x in t]
    assert not bad
