"""Exact medians with many classes, whose histograms have 16-bit counters from 12
classes on while a block's slice, a quarter of the points, has at most 65535: at that
edge with every point of a slice in one bin (an even and an odd one), with more keys in
range than the list holds, and on both sides of the class count. Bit for bit a sort.
"""
import numpy as np
import pytest

from test_gpu_medians import _dev, _median, _values, env  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(env, V, n, seed):
    cs, ctx, torch = env
    k, N = V.shape
    init = np.random.default_rng(seed).choice(N, n, replace=False).astype(np.int32)
    Vd = _dev(torch, V)
    lab = ctx.kmedians(Vd, init, 0)["assign"].cpu().numpy()
    C = ctx.kmedians(Vd, init, 1)["centres"].cpu().numpy()
    ctx.sync()
    for b in range(n):
        mem = V[:, lab == b]
        want = np.array([_median(mem[j]) if mem.shape[1] else V[j, init[b]] for j in range(k)],
                        np.float32)
        np.testing.assert_array_equal(C[b], want)


@pytest.mark.parametrize("N", [262140, 262141])
@pytest.mark.parametrize("value", [1.0, 513.5 / 1024])  # bins 1920 and 1409
def test_one_bin(env, N, value):  # noqa: F811
    _check(env, np.full((1, N), value, np.float32), 12, 1)


@pytest.mark.parametrize("kind", ["iota", "wide", "two", "edges"])
@pytest.mark.parametrize("N,n", [(16, 16), (9001, 11), (9001, 12), (40001, 14), (262140, 12)])
def test_many_classes(env, kind, N, n):  # noqa: F811
    _check(env, _values(kind, np.random.default_rng(N + n), 2, N), n, n)
