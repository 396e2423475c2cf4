"""Which engine FP32 Jacobi and CG take (hs_last_quads): four nodes per lane or
one.  Values of tile_rows outside 4 .. 16 mean the same as 0.  Histories agree
between the engines to 1e-5 (the bar of the other FP32 CG comparison).  Chunks of
one to three planes run the quads' ring empty and full: Jacobi iterates stay
bitwise those of the one-node engine."""
import numpy as np
import pytest

from paper_2305_05988_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2305_05988_gb300 as hs  # noqa: E402
from paper_2305_05988_gb300 import _lib  # noqa: E402
from test_gpu_parity import dev  # noqa: E402

QUADS = [(64, 16, 128), (100, 37, 40), (252, 33, 19), (48, 64, 43), (64, 64, 32)]
# n_x not a multiple of 4; fewer than 2^17 nodes; tiles less than three quarters full
ONE = [(98, 37, 40), (64, 64, 31), (80, 41, 40), (44, 64, 48)]


@pytest.mark.parametrize("solver", ["cg", "jacobi"])
@pytest.mark.parametrize("rows", [0, 1, 3, 17, -1])
@pytest.mark.parametrize("shape", QUADS + ONE)
def test_engine(shape, rows, solver):
    A = hs.Operator.laplacian(shape)
    b = dev(inputs.uniform_pm1(91, 1, A.N), torch.float32)
    if solver == "cg":
        run = lambda **k: hs.cg(A, b, tol=0.0, maxit=6, **k)[1].history  # noqa: E731
    else:
        run = lambda **k: hs.jacobi(A, b, tol=1e-30, maxit=6, history=True, **k)[1].history  # noqa: E731
    h = run(tile_rows=rows)
    assert _lib.load().hs_last_quads() == (1 if shape in QUADS else 0)
    one = run(tile_rows=8)
    assert _lib.load().hs_last_quads() == 0
    assert np.allclose(h, one, rtol=1e-5, atol=0)


@pytest.mark.parametrize("planes", [1, 2, 3])
@pytest.mark.parametrize("shape", [(64, 16, 128), (100, 37, 40), (512, 129, 2)])
def test_short_chunks(shape, planes):
    A = hs.Operator.laplacian(shape)
    b = dev(inputs.uniform_pm1(92, 1, A.N), torch.float32)
    x, _ = hs.jacobi(A, b, maxit=5, tile_planes=planes)
    y, _ = hs.jacobi(A, b, maxit=5, tile_rows=8)
    assert torch.equal(x, y)
