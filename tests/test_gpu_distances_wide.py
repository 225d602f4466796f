"""The distance transform's column pass by the number of columns (labels x width): 8
columns per block and 6 segments (8 in tall narrow images), or 32 columns and 2 segments
(from 6000 columns on, at most 256 rows) or 4 (from 16000 on); at the edges of that rule
and of each form's shared memory (stacks of 440, 1758 and 1760 rows), with a last block
that is not full and rows that the segments don't share evenly: exact integers, equal to
the oracle's brute force.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,m", [
    (66, 5999, [2]),           # 8 columns, 6 segments
    (59, 6000, [5]),           # 32 columns, 2 segments
    (256, 3001, [1, 3]),
    (257, 3001, [1, 3]),       # 8 columns again
    (261, 15999, [4]),
    (261, 16001, [4]),         # 32 columns, 4 segments
    (440, 5347, [1, 1, 1]),    # the tallest in shared memory
    (441, 5347, [1, 1, 1]),
    (1536, 13, [3, 2]),        # 8 columns, 6 segments
    (1537, 13, [3, 2]),        # 8 segments
    (1758, 2001, [1, 2]),      # 6 segments, the tallest in shared memory
    (1759, 2001, [1, 2]),
])
def test_column_forms(cuda_lib, H, W, m):
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
