"""The neighbour-sum engine (FP64 operators with one coupling for all
neighbours) over the values it can meet: any exponents, cancelling and zero
neighbours, subnormals, infinities and NaNs, on shapes around the tile edges
(32 columns, 8 rows, chunks of planes) through SpMV and the residual.

Bound, derived before the first run: the neighbours are summed to within
7 * 2^-59 of the largest one and rounded once, then one FMA and (residual) one
more; with the roundings of the coefficients every node is within
8 * 2^-53 (|27 c| + sum |neighbours| [+ |b|]) of the exact value, plus one
subnormal spacing.  The reference is numpy's extended precision."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2305_05988_gb300 as hs  # noqa: E402

SHAPES = [(1, 1, 1), (2, 3, 4), (31, 9, 5), (32, 8, 33), (33, 7, 2), (34, 17, 70), (65, 16, 3), (40, 24),
          (33, 65), (1, 9, 40)]


def values(kind, N, rng):
    v = rng.uniform(-1, 1, N)
    if kind == "uniform":
        return v
    if kind == "wide":                       # neighbours 2^-300 .. 2^300 apart
        return np.ldexp(v, rng.integers(-300, 301, N))
    if kind == "cancel":                     # +-1 with last-place noise, many exact zeros of the sum
        return np.where(rng.random(N) < 0.5, 1.0, -1.0) * (1 + rng.integers(0, 3, N) * 2.0 ** -52)
    if kind == "sparse":
        return np.where(rng.random(N) < 0.05, v, 0.0)
    if kind == "tiny":                       # subnormals among small normals
        return np.ldexp(v, rng.integers(-1074, -1000, N))
    assert kind == "huge"
    return np.ldexp(v, rng.integers(900, 1014, N))


def neighbour_sums(x, shape):
    """Sum of the neighbours and of their magnitudes, in extended precision."""
    a = x.astype(np.longdouble).reshape(tuple(reversed(shape)))
    p = np.pad(a, 1)
    c = tuple(slice(1, -1) for _ in a.shape)
    s, m = np.zeros_like(a), np.zeros_like(a)
    for ax in range(a.ndim):
        for lo in (0, 2):
            q = p[c[:ax] + (slice(lo, lo + a.shape[ax]),) + c[ax + 1:]]
            s += q
            m += np.abs(q)
    return s.reshape(-1), m.reshape(-1)


@pytest.mark.parametrize("kind", ["uniform", "wide", "cancel", "sparse", "tiny", "huge"])
@pytest.mark.parametrize("shape", SHAPES)
def test_sum_within_bound(shape, kind):
    N = int(np.prod(shape))
    rng = np.random.default_rng(N + len(kind))
    x, b = values(kind, N, rng), values(kind, N, rng)
    A = hs.Operator.hpcg(shape, 7)
    s, m = neighbour_sums(x, shape)
    c = x.astype(np.longdouble)
    xt, bt = torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda()
    eps, sub = np.longdouble(8.0 * 2.0 ** -53), np.longdouble(2.0) ** -1073
    y = A.spmv(xt).cpu().numpy()
    assert np.all(np.abs(y - (27 * c - s)) <= eps * (27 * np.abs(c) + m) + sub)
    r = A.residual(bt, xt).cpu().numpy()
    assert np.all(np.abs(r - (b - (27 * c - s))) <= eps * (27 * np.abs(c) + m + np.abs(b)) + 2 * sub)


@pytest.mark.parametrize("shape", [(34, 17, 9), (33, 19)])
def test_non_finite_neighbours(shape):
    N = int(np.prod(shape))
    rng = np.random.default_rng(5)
    x = rng.uniform(-1, 1, N)
    at = rng.choice(N, 6, replace=False)
    x[at] = [np.inf, -np.inf, np.nan, np.inf, -np.inf, np.inf]
    y = hs.Operator.hpcg(shape, 7).spmv(torch.from_numpy(x).cuda()).cpu().numpy()
    with np.errstate(invalid="ignore"):
        s, _ = neighbour_sums(x, shape)
        ref = (27 * x.astype(np.longdouble) - s).astype(np.float64)
    assert np.array_equal(np.isnan(y), np.isnan(ref))
    assert np.array_equal(y[np.isinf(ref)], ref[np.isinf(ref)])
    fine = np.isfinite(ref)
    assert np.allclose(y[fine], ref[fine], rtol=1e-13, atol=1e-13)
