"""FP32 volume pass: dh/dt takes one rounding a term.  The rms error of dh/dt in units of 2^-24 of its terms'
magnitude (extended_residual.py), on fixed inputs with two and three nodes an element, against that of a pass whose
sums are taken term by term with fused multiply-adds (measured on the same inputs: the limits), within 1 %; a product
rounded apart from its sum costs 2 to 10 %.
"""
import numpy as np
import pytest

import extended_residual as X

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("p,rough,rms", [(1, 1.0, 0.0754), (1, 0.0, 0.0650), (2, 1.0, 0.0829), (2, 0.0, 0.0697)])
def test_depth_rate(p, rough, rms):
    import paper_2301_11238_gb300 as G
    K = 20000
    prm = dict(g=9.81, rho=1.0, alpha=0.05, eta=0.05, sigma0=0.0, gamma=1.0, beta=1.0, pap_m=1.0, h_floor=1e-6,
               cfl=0.3, reg=0, positivity=0)
    coords = np.linspace(0.0, 1.0, K + 1).reshape(-1, 1)
    etov = np.stack([np.arange(K), np.arange(1, K + 1)], 1).astype(np.int32)
    s = G.Solver(1, coords, etov, p, 0, prm, precision=G.PREC_FP32)
    x = s.node_coords()[..., 0]
    r = np.random.default_rng(p)
    noise = [rough * r.uniform(-1, 1, x.shape) for _ in range(2)]
    V = np.stack([1 + 0.2 * np.sin(4 * x + x) + 0.1 * noise[0], 0.3 * np.cos(4 * x) + 0.2 * noise[1]])
    V = V.astype(np.float32).astype(np.float64)
    dV = s.residual(V, with_E=False).cpu().numpy()
    ref, mag, _, _ = X.Rhs(coords, etov, p, prm).rate(V)
    err = float(np.sqrt(np.mean(((dV[0] - ref[0]) / mag[0]) ** 2))) * 2 ** 24
    assert err < 1.01 * rms, err
