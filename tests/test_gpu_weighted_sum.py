"""Weighted neighbour sums (FP64) with couplings far apart: every axis as the
weak one, ratios just inside the rule (62 in 3-D and 2-D) and just outside (81,
the general path), values that lie along the weak axis or across it.

Bound, derived before the first run: a coupling relative to the upper x one is
rounded once, the sum is within 7.5 x 2^-56 of the largest weighted term before
its one rounding, then one FMA with the rounded diagonal and the scaling: at
most 6 x 2^-53 of |d c| + sum |a_q x_q| with second-order terms.  Outside the
rule the couplings' chain of FMAs rounds six times instead: 11 x 2^-53.  The
reference is numpy's extended precision."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_neighbour_sum import neighbour_sums, operator  # noqa: E402

INSIDE = [(62, 62, 7), (62, 7, 62), (7, 62, 62), (62, 7), (7, 62), (46, 46, 5)]
OUTSIDE = [(71, 71, 7), (7, 71)]


def values(kind, shape, rng):
    """Large values on every other plane across the weak axis; between them
    zeros ("only"), values 2^-6 .. 2^-20 of them ("small"), or the reverse
    ("across": the planes' own values are large, so the strong axes' are)."""
    weak = int(np.argmin(shape))
    at = np.indices(tuple(reversed(shape)))[len(shape) - 1 - weak].reshape(-1)
    v = rng.uniform(-1, 1, at.size)
    if kind == "only":
        return np.where(at % 2 == 1, v, 0.0)
    small = np.ldexp(v, -rng.integers(6, 21, at.size))
    return np.where(at % 2 == (1 if kind == "small" else 0), v, small)


@pytest.mark.parametrize("kind", ["only", "small", "across"])
@pytest.mark.parametrize("op", ["laplacian", "upwind"])
@pytest.mark.parametrize("shape", INSIDE + OUTSIDE)
def test_couplings_far_apart(shape, op, kind):
    rng = np.random.default_rng(sum(shape) + len(kind))
    x = values(kind, shape, rng)
    A, d, lo, up = operator(op, shape)
    s, m = neighbour_sums(x, shape, lo, up)
    c = x.astype(np.longdouble) * np.longdouble(d)
    y = A.spmv(torch.from_numpy(x).cuda()).cpu().numpy()
    r = A.residual(torch.zeros(x.size, dtype=torch.float64, device="cuda"), torch.from_numpy(x).cuda()).cpu().numpy()
    eps = np.longdouble((6.0 if shape in INSIDE else 11.0) * 2.0 ** -53)
    assert np.all(np.abs(y - (c - s)) <= eps * (np.abs(c) + m))
    assert np.all(np.abs(r + (c - s)) <= eps * (np.abs(c) + m))
