"""Jacobi sweeps on 2-D grids on both sides of the size at which weighted
neighbour sums give way to the general form (7 x 2^19 nodes), against plain
PyTorch sweeps in FP64 (1e-12, the bar of the other Jacobi comparisons)."""
import pytest

from paper_2305_05988_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2305_05988_gb300 as hs  # noqa: E402


@pytest.mark.parametrize("op", ["laplacian", "upwind"])
@pytest.mark.parametrize("shape", [(2048, 1792), (2049, 1792), (1900, 1933)])
def test_sweeps(shape, op):
    nx, ny = shape
    beta = inputs.upwind_beta(shape, 0.5) if op == "upwind" else (0.0, 0.0)
    A = hs.Operator.upwind(shape, beta) if op == "upwind" else hs.Operator.laplacian(shape)
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    b = torch.rand(A.N, dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    x0 = torch.rand(A.N, dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    x, _ = hs.jacobi(A, b, x0, maxit=3)
    up = [float((n + 1) ** 2) for n in shape]
    lo = [u + beta[q] * (shape[q] + 1) for q, u in enumerate(up)]
    d = sum(up) + sum(lo)
    r, bb = x0.reshape(ny, nx), b.reshape(ny, nx)
    for _ in range(3):
        p = torch.nn.functional.pad(r, (1, 1, 1, 1))
        r = (bb + lo[0] * p[1:-1, :-2] + up[0] * p[1:-1, 2:] + lo[1] * p[:-2, 1:-1] + up[1] * p[2:, 1:-1]) / d
    assert ((x.reshape(ny, nx) - r).norm() / r.norm()).item() <= 1e-12
