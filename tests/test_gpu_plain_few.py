"""The plain FP32 sum's form for few samples per label: code counts by words, samples
around its groups of 16 and its 64-sample tiles, pixels around its blocks of 128, both
sides of the rule that picks it (60000 pixels; 40 pixels a padded sample; 192 padded
samples a label, fewer with more than four words), and pixel lists (the surrogate's
targets and fallback). Bar: the plain form's 1e-5 relative on L against the FP64 oracle; a
wrong TSM by one moves L by more than 1e-3.
"""
import numpy as np
import pytest

from paper_1312_4746_gb300 import synth
from test_gpu_plain_sum import _check, _dev, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 31, 32, 33, 98, 128, 160, 192, 224, 256])
@pytest.mark.parametrize("mode", [0, 1])
def test_code_counts(env, k, mode):  # noqa: F811
    _check(env, synth.make_problem(61, 83, 3, [10, 15, 30], p=5, k=k, seed=800 + k, cap_frac=0.9),
           mode)


@pytest.mark.parametrize("m", [[1], [15, 16], [17, 64], [65, 48], [2, 100]])
@pytest.mark.parametrize("mode", [0, 1])
def test_sample_counts(env, m, mode):  # noqa: F811
    _check(env, synth.make_problem(80, 90, len(m), m, p=3, k=18, seed=820 + m[0], cap_frac=0.9), mode)


@pytest.mark.parametrize("H,W", [(1, 639), (1, 640), (1, 641), (769, 1), (7, 128)])  # rule: 16 x 40
def test_pixel_counts(env, H, W):  # noqa: F811
    _check(env, synth.make_problem(H, W, 1, 9, p=3, k=40, seed=840 + W, cap_frac=0.9), 0)


@pytest.mark.parametrize("H,W,m,k", [
    (199, 301, [192, 190], 40), (200, 300, [192, 190], 40), (200, 300, [193, 190], 40),
    (200, 300, [128, 120], 162), (200, 300, [128, 129], 162),
    (152, 257, [400, 5, 64, 430], 50),  # general, two operand tiles per block
])
@pytest.mark.parametrize("mode", [0, 1])
def test_rule(env, H, W, m, k, mode):  # noqa: F811
    pr = synth.make_problem(H, W, len(m), m, p=5, k=k, seed=860 + k)
    pix = np.unique(np.random.default_rng(2).integers(0, H * W, 1500)).astype(np.int32)
    _check(env, pr, mode, pix)


@pytest.mark.parametrize("mode", [0, 1])
def test_pixel_lists(env, mode):  # noqa: F811
    cs, ctx, torch = env
    pr = synth.make_problem(70, 90, 3, [9, 20, 33], p=5, k=50, seed=880)
    prm = cs.Params.from_synth(pr.params, mode=mode)
    img, om, mk, smp = (_dev(torch, a) for a in (pr.image, pr.omega, pr.mask, pr.sample_pix))
    cd = ctx.codes(img, om, mk, prm, want_lead16=True)
    args = (img, cd["bitmask"], cd["lead16"], 50, pr.label_off, smp, prm)
    want = ctx.likelihood(img, cd["bitmask"], 50, pr.label_off, smp, prm)
    ctx.surrogate_fit(*args, frac=0.2, steps=5)
    out, n = ctx.surrogate_eval(*args, margin=1.0, rule=cs.FALLBACK_MARGIN)  # every pixel
    ctx.sync()
    assert n == 70 * 90
    assert torch.equal(out["neglog"], want["neglog"]) and torch.equal(out["post"], want["post"])
