"""k-means centroids are exact: float32(S / (count 2^24)) with S the integer sum of
rint(2^24 v) over the members, whichever way a warp's members are added up (few
classes in the warp: each class's first; many: one by one; values of 2 and above one
by one as well). Compared bit for bit after one round.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 6, 7, 16])
@pytest.mark.parametrize("N", [31, 5000])
@pytest.mark.parametrize("lo,hi", [(0.0, 1.0), (-3.0, 9.0)])
def test_centroids_exact(cuda_lib, n, N, lo, hi):
    import torch

    import paper_1312_4746_gb300 as cs

    rng = np.random.default_rng(50 + n + N)
    X = rng.uniform(lo, hi, (N, 3)).astype(np.float32)
    X[N // 3:N // 2] = X[0]  # a stretch of one class
    init = rng.choice(np.arange(N // 2, N), n, replace=False).astype(np.int32) if n <= N // 2 \
        else np.arange(n, dtype=np.int32)
    ctx = cs.Context(0)
    Xd = torch.from_numpy(X).to("cuda:0")
    lab = ctx.kmeans(Xd, init, 0)["assign"].cpu().numpy()
    C = ctx.kmeans(Xd, init, 1)["centres"].cpu().numpy()
    ctx.sync()
    ctx.close()
    q = np.rint(X * np.float32(2 ** 24)).astype(np.int64)  # the product is exact
    for b in range(n):
        mem = lab == b
        want = (q[mem].sum(0).astype(np.float64) / (mem.sum() * 2.0 ** 24)).astype(np.float32) \
            if mem.any() else X[init[b]]
        np.testing.assert_array_equal(C[b], want)
