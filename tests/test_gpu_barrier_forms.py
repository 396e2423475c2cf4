"""BiCGStab on both sides of the team size at which its reduce-barrier changes
form (400 blocks), and with all blocks: the same iterates up to the order of the
sums (oracle, 5 iterations, 1e-11), repeated runs bitwise equal."""
import numpy as np
import pytest

import oracle
from paper_2305_05988_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2305_05988_gb300 as hs  # noqa: E402
from test_gpu_parity import dev, host, rel  # noqa: E402

SHAPE = (128, 120, 64)   # 1024 items of 4 planes


@pytest.mark.parametrize("blocks", [399, 400, 401, 0])
def test_bicgstab_team_sizes(blocks):
    beta = inputs.upwind_beta(SHAPE, 0.5)
    A, A_o = hs.Operator.upwind(SHAPE, beta), oracle.Operator(SHAPE, oracle.UPWIND, beta)
    b = inputs.uniform_pm1(81, 1, A.N)
    kw = dict(tol=0.0, maxit=5, tile_planes=4, max_blocks=blocks)
    x, i = hs.bicgstab(A, dev(b), **kw)
    y, j = hs.bicgstab(A, dev(b), **kw)
    assert i.iters == 5 and torch.equal(x, y) and np.array_equal(i.history, j.history)
    assert rel(host(x), oracle.bicgstab(A_o, b, tol=0.0, maxit=5)[0]) <= 1e-11
