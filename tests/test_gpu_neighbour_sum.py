"""The neighbour-sum engine (FP64 operators, equal or weighted couplings) over
the values it can meet: any exponents, cancelling and zero neighbours,
subnormals, infinities and NaNs, on shapes around the tile edges (32 columns,
8 rows, chunks of planes) through SpMV and the residual.

Bound, derived before the first run: the neighbours are summed to within
7 * 2^-59 (weighted: 6 * 2^-57) of the largest term and rounded once, then one
FMA, the scaling and (residual) one more; with the roundings of the scaled
coefficients (two each) every node is within
8 * 2^-53 (|d c| + sum |a_q x_q| [+ |b|]) of the exact value, plus a few
subnormal spacings times the scaling.  The reference is numpy's extended
precision.  A spacing ratio above 8 takes the general path."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2305_05988_gb300 as hs  # noqa: E402
from paper_2305_05988_gb300 import inputs  # noqa: E402

SHAPES = [(1, 1, 1), (2, 3, 4), (31, 9, 5), (32, 8, 33), (33, 7, 2), (34, 17, 70), (65, 16, 3), (40, 24),
          (33, 65), (1, 9, 40), (200, 10, 12)]


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


def operator(op, shape):
    """The operator and its couplings (diagonal, lower and upper per axis)."""
    nd = len(shape)
    if op == "hpcg7":
        return hs.Operator.hpcg(shape, 7), 27.0, [1.0] * nd, [1.0] * nd
    beta = inputs.upwind_beta(shape, 0.5) if op == "upwind" else (0.0,) * 3
    A = hs.Operator.upwind(shape, beta) if op == "upwind" else hs.Operator.laplacian(shape)
    h = [1.0 / (n + 1) for n in shape]
    up = [1.0 / (v * v) for v in h]
    lo = [u + beta[q] / h[q] for q, u in enumerate(up)]
    return A, sum(up) + sum(lo), lo, up


def neighbour_sums(x, shape, lo, up):
    """Weighted sum of the neighbours and of the terms' magnitudes, in extended precision."""
    a = x.astype(np.longdouble).reshape(tuple(reversed(shape)))
    p = np.pad(a, 1)
    c = tuple(slice(1, -1) for _ in a.shape)
    s, m = np.zeros_like(a), np.zeros_like(a)
    for ax in range(a.ndim):
        for at, w in ((0, lo), (2, up)):
            q = p[c[:ax] + (slice(at, at + a.shape[ax]),) + c[ax + 1:]] * np.longdouble(w[a.ndim - 1 - ax])
            s += q
            m += np.abs(q)
    return s.reshape(-1), m.reshape(-1)


@pytest.mark.parametrize("kind", ["uniform", "wide", "cancel", "sparse", "tiny", "huge"])
@pytest.mark.parametrize("op", ["hpcg7", "laplacian", "upwind"])
@pytest.mark.parametrize("shape", SHAPES)
def test_sum_within_bound(shape, op, kind):
    N = int(np.prod(shape))
    rng = np.random.default_rng(N + len(kind))
    x, b = values(kind, N, rng), values(kind, N, rng)
    A, d, lo, up = operator(op, shape)
    s, m = neighbour_sums(x, shape, lo, up)
    c = x.astype(np.longdouble) * np.longdouble(d)
    xt, bt = torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda()
    eps, sub = np.longdouble(8.0 * 2.0 ** -53), np.longdouble(2.0) ** -1073 * (1 + max(lo) + max(up)) * 4
    size = np.abs(c) + m + np.abs(b)
    fits = size < np.longdouble(2.0) ** 1023        # beyond, binary64 itself overflows
    y = A.spmv(xt).cpu().numpy()
    r = A.residual(bt, xt).cpu().numpy()
    with np.errstate(invalid="ignore"):
        ey, er = np.abs(y - (c - s)), np.abs(r - (b - (c - s)))
    assert np.all(ey[fits] <= (eps * (np.abs(c) + m) + sub)[fits])
    assert np.all(er[fits] <= (eps * size + 2 * sub)[fits])


@pytest.mark.parametrize("op", ["hpcg7", "laplacian", "upwind"])
@pytest.mark.parametrize("shape", [(34, 17, 9), (33, 19)])
def test_non_finite_neighbours(shape, op):
    N = int(np.prod(shape))
    rng = np.random.default_rng(5)
    x = rng.uniform(-1, 1, N)
    at = rng.choice(N, 6, replace=False)
    x[at] = [np.inf, -np.inf, np.nan, np.inf, -np.inf, np.inf]
    A, d, lo, up = operator(op, shape)
    y = A.spmv(torch.from_numpy(x).cuda()).cpu().numpy()
    with np.errstate(invalid="ignore"):
        s, m = neighbour_sums(x, shape, lo, up)
        ref = (np.longdouble(d) * x.astype(np.longdouble) - s).astype(np.float64)
    assert np.array_equal(np.isnan(y), np.isnan(ref))
    assert np.array_equal(y[np.isinf(ref)], ref[np.isinf(ref)])
    fine = np.isfinite(ref)
    assert np.all(np.abs(y[fine] - ref[fine]) <= 1e-15 * (np.abs(d * x[fine]) + m[fine].astype(np.float64)))
