"""Kernel forms that a single context takes by mesh size, each against the direct forms of a batch (block sizes set to
one thread per element and face point), just below and just above its line:

  FP32 p >= 2   faces in a grid-stride loop from 38,912 faces; p = 3 E-step in one from 38,912 elements
  FP64 p >= 2   faces in a grid-stride loop from 311,296 faces
  FP64          E-step with a thread per velocity component, volume pass in lanes, up to 9,728 elements

Sizes are ragged (no multiple of a block or of the grid); walls, copies and prescribed values at the boundary.  FP64
forms do the same operations: equal bit for bit.  FP32: 1e-6 relative L2 after two steps, 16 roundings of 6e-8.
"""
import numpy as np
import pytest

import synth
from helpers import rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def compare(nx, ny, p, precision):
    import paper_2301_11238_gb300 as G
    c = synth.radial_dam_2d(n=2, order=p, gamma=1.0)
    coords, etov = synth.rect_tri_mesh(nx, ny, jitter=0.1, seed=nx)
    K, faces = len(etov), 3 * nx * ny + nx + ny
    tags = (np.arange(3 * K).reshape(K, 3) % 3).astype(np.int8)
    bcs = [([0] * 7, [0.0] * 7), ([0, 2, 2, 0, 0, 0, 0], [0.0] * 7),
           ([1, 1, 1, 1, 1, 0, 0], [1.1, 0.2, -0.1, 0.3, 0.1, 0, 0])]
    spec = dict(dim=2, coords=coords, etov=etov, order=p, reg=c.params["reg"], prm=c.params, face_bc=tags, bcs=bcs)
    s = G.Solver(2, coords, etov, p, c.params["reg"], c.params, face_bc=tags, bcs=bcs, precision=precision)
    x = s.node_coords()
    V = np.stack([1 + 0.2 * np.sin(5 * x[..., 0] + x[..., 1]), 0.3 * np.cos(4 * x[..., 1]), 0.2 * np.sin(3 * x[..., 0])])
    b = G.Batch([spec], precision=precision)
    b.set_tiles([[128, 128, 128]])
    s.set_state(V)
    b.set_state(0, V)
    s.advance(2)
    b.advance(2)
    return K, faces, s.get_state(with_E=False), b.get_state(0), V


@pytest.mark.parametrize("nx,ny,above", [(113, 114, False), (114, 115, True)])
@pytest.mark.parametrize("p", [2, 3])
def test_fp32_faces(nx, ny, above, p):
    _, faces, V, W, V0 = compare(nx, ny, p, 1)
    assert (faces >= 38912) == above
    assert rel_l2(V, W) < 1e-6 and rel_l2(V, V0) > 1e-6


@pytest.mark.parametrize("nx,ny,above", [(139, 139, False), (139, 141, True)])
def test_fp32_estep(nx, ny, above):
    K, _, V, W, V0 = compare(nx, ny, 3, 1)
    assert (K >= 38912) == above
    assert rel_l2(V, W) < 1e-6 and rel_l2(V, V0) > 1e-6


@pytest.mark.parametrize("nx,ny,above", [(321, 322, False), (322, 323, True)])
@pytest.mark.parametrize("p", [2, 3])
def test_fp64_faces(nx, ny, above, p):
    _, faces, V, W, _ = compare(nx, ny, p, 0)
    assert (faces >= 311296) == above
    assert np.array_equal(V, W)


@pytest.mark.parametrize("nx,ny,lanes", [(65, 73, True), (64, 76, True), (67, 73, False)])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_fp64_estep_by_component(nx, ny, lanes, p):
    K, _, V, W, _ = compare(nx, ny, p, 0)
    assert (K <= 9728) == lanes
    assert np.array_equal(V, W)
