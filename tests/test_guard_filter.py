"""The guard pass's eight-lane filter (csrc/k_codes.cu, codes_guard_kernel): its
evaluation of a code (sums over eight lanes, lane l holding elements l, l + 8,
..., then a butterfly; the dot product taken before the one quotient) lies within
the bound that test_guard_bound.py checks for the index-order evaluation, with A
replaced by sqrt(N (ss + N mu^2)) >= sum |v_t|, of a 60-digit value; so a value
clear of tau by four times the bound decides the bit the index order decides.
"""
import math
from decimal import Decimal

import numpy as np
import pytest

from test_guard_bound import U, exact_code


def lane_sum(xs):
    lanes = [0.0] * 8
    for t, x in enumerate(xs):
        lanes[t % 8] = lanes[t % 8] + x
    o = 4
    while o:
        lanes = [lanes[l] + lanes[l ^ o] for l in range(8)]
        o >>= 1
    assert len(set(lanes)) == 1
    return lanes[0]


def filter_code(v, o):
    n = len(v)
    mu = lane_sum(v) * (1.0 / n)
    c = [x - mu for x in v]
    ss = lane_sum([x * x for x in c])  # (the kernel's fused products round less)
    nrm = math.sqrt(ss)
    es = 2 * U * n * math.sqrt(ss + n * mu * mu) / nrm + (0.5 * n + 5) * U
    return lane_sum([a * b for a, b in zip(o, c)]) / nrm, es, mu, ss


@pytest.mark.parametrize("n", [9, 25, 49, 81])
def test_filter_within_bound(n):
    rng = np.random.default_rng(100 + n)
    worst = 0.0
    for _ in range(60):
        base, spread = rng.uniform(0, 1), 10.0 ** rng.uniform(-7, 0)
        w = np.exp(-rng.uniform(0, 2, n))
        v = [float(x) for x in w * (base + spread * rng.standard_normal(n))]
        o = rng.standard_normal(n)
        o = [float(x) for x in (o / np.linalg.norm(o)).astype(np.float32)]
        a, es, mu, ss = filter_code(v, o)
        assert sum(abs(x) for x in v) <= math.sqrt(n * (ss + n * mu * mu)) * (1 + 1e-12)
        on = math.sqrt(sum(x * x for x in o))
        eps = on * (es + n * U * (1 + es))
        err = float(abs(Decimal(a) - exact_code(v, o)))
        assert err <= eps, (err, eps)
        worst = max(worst, err / eps)
    print(f"n = {n}: worst error / bound {worst:.3f}")
