"""lead16 is zero beyond the k codes of an operator with fewer than 16 rows, also at
pixels whose patch holds a NaN or an infinity, in both codes forms.
"""
import numpy as np
import pytest

from paper_1312_4746_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,k", [(3, 1), (5, 9), (9, 15), (7, 16)])
@pytest.mark.parametrize("form", [1, 2])  # CODES_FP32, CODES_TC
def test_zero_beyond_k(cuda_lib, p, k, form):
    import torch

    import paper_1312_4746_gb300 as cs

    pr = synth.make_problem(20, 37, 2, 5, p=p, k=k, seed=40 + k)
    image = pr.image.copy()
    image[3, 5, 1], image[15, 30, 0] = np.nan, np.inf
    ctx = cs.Context(0)
    img, om, mask = (torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
                     for a in (image, pr.omega, pr.mask))
    prm = cs.Params.from_synth(pr.params, codes_form=form)
    lead = ctx.codes(img, om, mask, prm, want_lead16=True)["lead16"].cpu().numpy()
    ctx.sync()
    ctx.close()
    assert not np.isfinite(lead[:, :k]).all()  # the codes themselves are not finite there
    assert np.array_equal(lead[:, k:], np.zeros_like(lead[:, k:]))
