"""The FP32 engine with four nodes per lane against the one-node engine
(tile_rows selects it) and the FP64 oracle, on shapes around its tile edges
(64 x 16 nodes, chunks of planes).

Every node runs the same arithmetic in both engines, so Jacobi iterates are
bitwise equal; CG's dot products are summed in another order, so its early
iterates agree to 1e-5 (the bar of the other FP32 CG comparison).  Oracle: a
sweep rounds at most 11 times at 2^-24, so k sweeps stay within 11 k 2^-24."""
import numpy as np
import pytest

import oracle
from paper_2305_05988_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2305_05988_gb300 as hs  # noqa: E402
from test_gpu_parity import dev, host, rel  # noqa: E402

# 2^17 nodes and more: whole tiles; ragged rows and columns; one plane more
# than a chunk; two planes; a last tile of one quad row
SHAPES = [(64, 16, 128), (100, 37, 40), (64, 17, 125), (252, 33, 19), (512, 129, 2), (116, 113, 11)]


def operators(shape, kind):
    if kind == "lap":
        return hs.Operator.laplacian(shape), oracle.Operator(shape)
    if kind == "up":
        beta = inputs.upwind_beta(shape, 0.5)
        return hs.Operator.upwind(shape, beta), oracle.Operator(shape, oracle.UPWIND, beta)
    k = np.exp(inputs.log_k(shape, 1.0, 3))
    return hs.Operator.diffusion(shape, dev(k)), oracle.Operator(shape, oracle.DIFFUSION, k=k)


@pytest.mark.parametrize("kind", ["lap", "up", "diff"])
@pytest.mark.parametrize("shape", SHAPES)
def test_jacobi(shape, kind):
    A, A_o = operators(shape, kind)
    b = inputs.uniform_pm1(71, 1, A.N)
    x0 = inputs.uniform_pm1(72, 1, A.N)
    bt, xt = dev(b, torch.float32), dev(x0, torch.float32)
    xq, _ = hs.jacobi(A, bt, xt, maxit=5)
    x1, _ = hs.jacobi(A, bt, xt, maxit=5, tile_rows=8)
    assert torch.equal(xq, x1)
    xo = oracle.jacobi(A_o, host(bt).astype(np.float64), host(xt).astype(np.float64), maxit=5)[0]
    assert rel(host(xq).astype(np.float64), xo) <= 5 * 11 * 2.0 ** -24
    # tolerance mode fuses the residual into the sweep
    xq, iq = hs.jacobi(A, bt, xt, tol=1e-30, maxit=4, history=True)
    x1, i1 = hs.jacobi(A, bt, xt, tol=1e-30, maxit=4, history=True, tile_rows=8)
    assert torch.equal(xq, x1) and np.allclose(iq.history, i1.history, rtol=1e-12, atol=0)


@pytest.mark.parametrize("kind", ["lap", "diff"])
@pytest.mark.parametrize("shape", SHAPES)
def test_cg(shape, kind):
    A, A_o = operators(shape, kind)
    b = inputs.uniform_pm1(73, 1, A.N)
    bt = dev(b, torch.float32)
    xq, iq = hs.cg(A, bt, tol=0.0, maxit=8)
    x1, i1 = hs.cg(A, bt, tol=0.0, maxit=8, tile_rows=8)
    assert iq.iters == i1.iters == 8
    assert rel(host(xq).astype(np.float64), host(x1).astype(np.float64)) <= 1e-5
    xo = oracle.cg(A_o, host(bt).astype(np.float64), tol=0.0, maxit=8)[0]
    assert rel(host(xq).astype(np.float64), xo) <= 1e-5
    assert np.allclose(iq.history, i1.history, rtol=1e-5, atol=0)
