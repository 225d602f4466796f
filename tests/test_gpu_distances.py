"""The distance transform's column passes at the edges of their rules (outward
scan up to labels x width x height^2 = 2e7 and 880 rows; envelopes of 2, 4 and 8
row segments, stacks in shared memory up to 1760 rows and in global memory
above), with columns that don't fill a block and segments without seeds: exact
integers, equal to the oracle's brute force.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,m", [
    (1, 23170, [1, 5]),        # scan, one row, the largest side
    (880, 25, [3]),            # scan, the tallest image
    (881, 25, [3, 1]),         # 8 segments
    (33, 9201, [2, 3]),        # 4 segments
    (32, 9799, [1, 40]),       # 2 segments
    (1760, 21, [1, 9]),        # 8 segments, the tallest image in shared memory
    (1761, 21, [1, 9]),        # 8 segments, stacks in global memory
    (23170, 3, [2]),           # the largest side, more readers than 8 segments share
])
def test_column_passes(cuda_lib, H, W, m):
    import torch

    import paper_1312_4746_gb300 as cs

    ctx = cs.Context(0)
    rng = np.random.default_rng(H + W)
    P = H * W
    smp = np.concatenate([np.sort(rng.choice(P, mi, replace=False)) for mi in m]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(m)]).astype(np.int32)
    dev = lambda a: torch.from_numpy(a).to("cuda:0")  # noqa: E731
    bits = torch.zeros((P, 1), dtype=torch.int32, device="cuda:0")
    img = dev(rng.uniform(0, 1, (H, W, 3)).astype(np.float32))
    out = ctx.likelihood(img, bits, 16, off, dev(smp), cs.Params.default(p=3), want_dist2=True)
    ctx.sync()
    assert np.array_equal(out["dist2"].cpu().numpy().reshape(len(m), -1),
                          oracle.dist2(H, W, off, smp))
    ctx.close()
