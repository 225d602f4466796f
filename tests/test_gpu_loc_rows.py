"""The tensor-core sum's location rows on both sides of the image size at which
their exact pieces change form (2880 pixels a side), and at tile remainders:
L within the derived recompute tolerance (l_tol 1e-4 relative) of the FP64
oracle at sampled pixels.
"""
import numpy as np
import pytest

import oracle
from paper_1312_4746_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,m", [(9, 2880, 300), (9, 2881, 300), (2880, 7, 256), (2881, 7, 129)])
@pytest.mark.parametrize("precision", [1, 2])
def test_loc_rows(cuda_lib, H, W, m, precision):
    import torch

    import paper_1312_4746_gb300 as cs

    ctx = cs.Context(0)
    pr = synth.make_problem(H, W, 2, m, p=3, k=18, seed=940 + W, cap_frac=0.9)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")  # noqa: E731
    prm = cs.Params.from_synth(pr.params, precision=precision)
    prm.l_tol = 1e-4
    out = ctx.data_term(dev(pr.image), dev(pr.omega), dev(pr.mask), pr.label_off,
                        dev(pr.sample_pix), prm)
    ctx.sync()
    pix = np.unique(np.random.default_rng(2).integers(0, H * W, 1500)).astype(np.int32)
    L = -out["neglog"].cpu().numpy().reshape(2, -1)[:, pix].astype(np.float64)
    ref = oracle.data_term(pr, pix=pix)["L"]
    assert np.max(np.abs(L - ref) / np.maximum(np.abs(ref), 1.0)) <= 1e-4
    ctx.close()
