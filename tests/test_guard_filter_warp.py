"""The guard pass's filter with a whole warp per entry (csrc/k_codes.cu, short lists):
as test_guard_filter.py with sums over 32 lanes, lane l holding elements l, l + 32, ...,
then a butterfly.
"""
from decimal import Decimal

import numpy as np
import pytest

import test_guard_filter
from test_guard_bound import U, exact_code


def lane_sum32(xs):
    lanes = [0.0] * 32
    for t, x in enumerate(xs):
        lanes[t % 32] = lanes[t % 32] + x
    o = 16
    while o:
        lanes = [lanes[l] + lanes[l ^ o] for l in range(32)]
        o >>= 1
    assert len(set(lanes)) == 1
    return lanes[0]


@pytest.mark.parametrize("n", [9, 25, 49, 81])
def test_filter_within_bound(n, monkeypatch):
    monkeypatch.setattr(test_guard_filter, "lane_sum", lane_sum32)
    rng = np.random.default_rng(300 + n)
    for _ in range(60):
        base, spread = rng.uniform(0, 1), 10.0 ** rng.uniform(-7, 0)
        w = np.exp(-rng.uniform(0, 2, n))
        v = [float(x) for x in w * (base + spread * rng.standard_normal(n))]
        o = rng.standard_normal(n)
        o = [float(x) for x in (o / np.linalg.norm(o)).astype(np.float32)]
        a, es, _, _ = test_guard_filter.filter_code(v, o)
        on = float(np.sqrt(sum(x * x for x in o)))
        assert float(abs(Decimal(a) - exact_code(v, o))) <= on * (es + n * U * (1 + es))
