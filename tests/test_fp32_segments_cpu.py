"""The arithmetic of the FP32 CUDA-core Legendre kernels, simulated on the CPU (no
GPU): a segment of 32 degrees starts from the FP64 state, stored as it is when
it is at least 2^-63, else times the power of two that takes the segment's
largest value to about 2^50, with the factor that takes it back; segments whose
values are all below 2^-70 are left out.  Every operation is rounded to FP32,
subnormals included.

1. The error of P, by the measure of test_fp32_recurrence_cpu.py (which simulates
   an exponent counter per value, a form the kernels no longer have): within
   B_F32_REC, the constant that the GPU parity tests rest on.
2. Sums over latitudes of P times small data (folds of 2^-97: a grid of 2^-80 times
   quadrature weights near 2^-17) are as exact as those of O(1) data: the factor
   multiplies P.  Multiplied into the folds instead it loses ordinary terms."""
import math

import numpy as np
import pytest

import oracle
from _bounds import B_F32_REC

SEG, TOP, LEAST, ASIS = 32, 50, -70, -63
FOLD = 2.0 ** -97
# truncation, sampled orders: from the poles' smooth orders to those that start far
# below the FP32 range almost everywhere
CASES = [(1023, (0, 10, 100, 400, 800, 1000)), (2047, (1400, 1900, 2040))]


def f32(v):
    with np.errstate(under="ignore", over="ignore"):
        return np.asarray(v, dtype=np.float64).astype(np.float32).astype(np.float64)


def coefficients(lmax, m):
    n = np.arange(m, lmax + 1, dtype=np.float64)
    a, b = np.zeros_like(n), np.zeros_like(n)
    b[0] = 1.0          # the start value, handed over as P_{m-2}
    if len(n) > 1:
        a[1] = math.sqrt(2 * m + 3)
    k = n[2:]
    a[2:] = np.sqrt((4 * k * k - 1) / (k * k - m * m))
    b[2:] = -np.sqrt((2 * k + 1) / (2 * k - 3) * ((k - 1) ** 2 - m * m) / (k * k - m * m))
    return f32(a), f32(b)


def exponent(v):
    """floor(log2 |v|), far below everything for 0."""
    return np.where(v == 0, -5000, np.frexp(v)[1] - 1)


def segment_states(true, s):
    """(y1, y2, factor) per node of the segment s of an order, from its exact values [degree, node]."""
    i0 = SEG * s
    zero = np.zeros(true.shape[1])
    t1, t2 = (zero, true[0]) if s == 0 else (true[i0 - 1], true[i0 - 2])
    top = exponent(np.abs(true[i0:i0 + SEG]).max(axis=0))
    h = np.maximum(exponent(t1), exponent(t2))
    e = np.where(h >= ASIS, 0, TOP - top)
    none = (h <= -1022) | (top < LEAST)
    with np.errstate(over="ignore"):
        y1, y2 = (np.where(none, 0.0, f32(np.ldexp(t, np.where(none, 0, e)))) for t in (t1, t2))
    return y1, y2, np.where(none, 0.0, np.ldexp(1.0, -np.where(none, 0, e)))


def segment(ab, x, y1, y2):
    """The recurrence in FP32: rows of y, P = factor y."""
    out = []
    for a, b in zip(*ab):
        y1, y2 = f32(f32(a * x) * y1 + f32(b * y2)), y1     # a fused multiply-add of rounded products
        out.append(y1)
    return np.array(out)


def order_values(lmax, m, x, true):
    """[degree, node] y, and factor [segment, node]."""
    a, b = coefficients(lmax, m)
    rows, fac = [], []
    for s in range((lmax - m + SEG) // SEG):
        y1, y2, f = segment_states(true, s)
        d = slice(SEG * s, SEG * (s + 1))
        rows.append(segment((a[d], b[d]), f32(x), y1, y2))
        fac.append(f)
    return rows, fac


@pytest.fixture(scope="module", params=[(n, m) for n, ms in CASES for m in ms], ids=lambda v: f"N{v[0]}-m{v[1]}")
def order(request):
    lmax, m = request.param
    nlat = lmax + 1
    x = oracle.gauss(nlat)[0][: nlat // 2][:: max(1, nlat // 1024)]
    true = oracle.plm_order(lmax, m, x).T
    return lmax, m, x, true, order_values(lmax, m, x, true)


def test_values_within_the_constant(order):
    _, _, _, true, (rows, fac) = order
    y = np.concatenate(rows)
    assert np.isfinite(y).all() and np.abs(y).max() < 2.0 ** 100
    f = np.concatenate([np.broadcast_to(v, r.shape) for v, r in zip(fac, rows)])
    assert ((f == 0) | (f >= 2.0 ** -126)).all()            # a normal number
    got = f32(f * y)
    rss = np.sqrt((true ** 2).sum(axis=0))
    live = rss >= 1e-7 * rss.max()
    err = np.sqrt(((got - true) ** 2).sum(axis=0))
    assert (err[live] / rss[live]).max() <= B_F32_REC


def test_sums_of_small_data(order):
    """Sums over the nodes, degree by degree, by fused multiply-adds in the nodes'
    order; the error over the root of the sum of the terms' squares.  The bound is
    that of O(1) data: half of B_F32_REC for P (its measure, over random data) and
    a rounding of 2^-24 per addition, at random."""
    _, _, x, true, (rows, fac) = order
    fold = f32(np.random.default_rng(1).standard_normal(len(x)) * FOLD)
    bad = False
    for s, (y, f) in enumerate(zip(rows, fac)):
        t = true[SEG * s:SEG * (s + 1)]
        terms = np.sqrt(((t * fold) ** 2).sum(axis=1))
        exact = (t * fold).sum(axis=1)
        keep = terms >= FOLD * 2.0 ** -30             # not the orders' vanishing starts
        acc, was = np.zeros(len(t)), np.zeros(len(t))
        for j in range(len(x)):
            acc = f32(acc + f32(f[j] * y[:, j]) * fold[j])
            was = f32(was + y[:, j] * f32(f[j] * fold[j]))
        bound = (B_F32_REC + 2.0 ** -24 * math.sqrt(len(x))) * terms
        assert (np.abs(acc - exact) <= bound)[keep].all()
        bad = bad or (np.abs(was - exact) > bound)[keep].any()
    if (np.concatenate(fac) < 2.0 ** -30).any() and (np.concatenate(fac) > 0).any():
        order_scaled.append((order[0], order[1], bad))


order_scaled = []


def test_factor_in_the_data_would_lose_terms():
    """Some of the sampled orders show it (those with a scaled segment that reaches O(1))."""
    assert any(b for _, _, b in order_scaled)
