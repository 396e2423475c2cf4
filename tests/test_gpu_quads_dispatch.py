"""Which engine FP32 Jacobi and CG take.  The quads (64 x 16 nodes per block) sum
their dot products in another order than the one-node engine, so a residual
history is bitwise that of tile_rows = 8 exactly where the one-node engine (8
rows on 3-D grids) ran.  Values of tile_rows outside 4 .. 16 mean the same as 0.
Chunks of one to three planes run the quads' ring empty and full: Jacobi
iterates stay bitwise those of the one-node engine."""
import numpy as np
import pytest

from paper_2305_05988_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2305_05988_gb300 as hs  # noqa: E402
from test_gpu_parity import dev  # noqa: E402

QUADS = [(64, 16, 128), (100, 37, 40), (252, 33, 19), (48, 64, 43), (64, 64, 32)]
# n_x not a multiple of 4; fewer than 2^17 nodes; tiles less than three quarters full
ONE = [(98, 37, 40), (64, 64, 31), (80, 41, 40), (44, 64, 48)]


def histories(shape, solver, **kw):
    A = hs.Operator.laplacian(shape)
    b = dev(inputs.uniform_pm1(91, 1, A.N), torch.float32)
    run = (lambda **k: hs.cg(A, b, tol=0.0, maxit=6, **k)) if solver == "cg" else \
        (lambda **k: hs.jacobi(A, b, tol=1e-30, maxit=6, history=True, **k))
    return run(**kw)[1].history, run(tile_rows=8)[1].history


@pytest.mark.parametrize("solver", ["cg", "jacobi"])
@pytest.mark.parametrize("rows", [0, 1, 3, 17, -1])
@pytest.mark.parametrize("shape", QUADS + ONE)
def test_engine(shape, rows, solver):
    h, one = histories(shape, solver, tile_rows=rows)
    assert np.allclose(h, one, rtol=1e-5, atol=0)
    assert np.array_equal(h, one) == (shape in ONE)


@pytest.mark.parametrize("planes", [1, 2, 3])
@pytest.mark.parametrize("shape", [(64, 16, 128), (100, 37, 40), (512, 129, 2)])
def test_short_chunks(shape, planes):
    A = hs.Operator.laplacian(shape)
    b = dev(inputs.uniform_pm1(92, 1, A.N), torch.float32)
    x, _ = hs.jacobi(A, b, maxit=5, tile_planes=planes)
    y, _ = hs.jacobi(A, b, maxit=5, tile_rows=8)
    assert torch.equal(x, y)
