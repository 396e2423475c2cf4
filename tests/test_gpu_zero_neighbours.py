"""Nodes whose neighbours are all zeros (the exit of the FP64 neighbour sums):
zeros of both signs, zeros next to subnormals and to ordinary values, through
SpMV in 2-D and 3-D with equal, unequal and upwind couplings.

A node with zeros all around is exactly d c; its sign of zero is that of
d c - s with s = -0 if every neighbour is -0 (outside the grid: +0), else +0.
Elsewhere the sum's bound of 8 x 2^-53 of the terms holds, with a few subnormal
spacings."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_neighbour_sum import neighbour_sums, operator  # noqa: E402


def values(kind, N, rng):
    zero = np.where(rng.random(N) < 0.5, 0.0, -0.0)
    if kind == "minus":
        return np.full(N, -0.0)
    if kind == "signs":
        return zero
    if kind == "points":                     # one node in 50 carries a value
        return np.where(rng.random(N) < 0.02, rng.uniform(-1, 1, N), zero)
    assert kind == "subnormal"
    return np.where(rng.random(N) < 0.3, rng.integers(-3, 4, N) * 5e-324, zero)


@pytest.mark.parametrize("kind", ["minus", "signs", "points", "subnormal"])
@pytest.mark.parametrize("op", ["hpcg7", "laplacian", "upwind"])
@pytest.mark.parametrize("shape", [(34, 17, 9), (33, 19), (40, 40)])
def test_zero_neighbours(shape, op, kind):
    N = int(np.prod(shape))
    x = values(kind, N, np.random.default_rng(N + len(kind)))
    A, d, lo, up = operator(op, shape)
    y = A.spmv(torch.from_numpy(x).cuda()).cpu().numpy()
    s, m = neighbour_sums(x, shape, lo, up)
    c = x.astype(np.longdouble) * np.longdouble(d)
    sub = np.longdouble(2.0) ** -1073 * (1 + max(lo) + max(up)) * 4
    assert np.all(np.abs(y - (c - s)) <= np.longdouble(8.0 * 2.0 ** -53) * (np.abs(c) + m) + sub)
    # nodes with zeros all around: the neighbours' signs, +0 outside the grid
    a = np.signbit(x.reshape(tuple(reversed(shape))))
    p = np.pad(a, 1, constant_values=False)
    core = tuple(slice(1, -1) for _ in shape)
    minus = np.ones_like(a)
    for ax in range(a.ndim):
        for at in (0, 2):
            minus &= p[core[:ax] + (slice(at, at + a.shape[ax]),) + core[ax + 1:]]
    ref = d * x - np.where(minus.reshape(-1), -0.0, 0.0)
    at = (m == 0) & (x == 0)
    assert np.all(y[at] == 0) and np.array_equal(np.signbit(y[at]), np.signbit(ref[at]))
