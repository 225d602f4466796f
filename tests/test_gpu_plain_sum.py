"""The plain FP32 sum at the edges of its layout: code counts around the 32-column
operand steps (the two columns of -|b_x| move into a step of their own), samples
around the 64-sample tiles and the 16-sample groups, pixels around the 128-pixel
operand tiles and on both sides of the rule that picks one or two of them per
CTA. Bar: the plain form's 1e-5 relative on L against the FP64 oracle; a wrong
TSM by one moves L by more than 1e-3.
"""
import numpy as np
import pytest

import oracle
from paper_1312_4746_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(cuda_lib):
    import torch

    import paper_1312_4746_gb300 as cs

    ctx = cs.Context(0)
    yield cs, ctx, torch
    ctx.close()


def _dev(torch, a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def _check(env, pr, mode, pix=None):
    cs, ctx, torch = env
    pr.params.mode = mode
    prm = cs.Params.from_synth(pr.params)
    out = ctx.data_term(_dev(torch, pr.image), _dev(torch, pr.omega), _dev(torch, pr.mask),
                        pr.label_off, _dev(torch, pr.sample_pix), prm)
    ctx.sync()
    L = -out["neglog"].cpu().numpy().reshape(pr.n_labels, -1).astype(np.float64)
    post = out["post"].cpu().numpy().reshape(pr.n_labels, -1)
    ref = oracle.data_term(pr, pix=pix)
    if pix is not None:
        L, post = L[:, pix], post[:, pix]
    assert np.max(np.abs(L - ref["L"]) / np.maximum(np.abs(ref["L"]), 1.0)) <= 1e-5
    assert np.max(np.abs(post - ref["post"])) <= 1e-4


@pytest.mark.parametrize("k", [1, 29, 30, 31, 32, 33, 62, 63, 94, 95, 126, 127, 128, 158, 190, 222,
                               223, 254, 255, 256])
def test_plain_code_counts(env, k):
    _check(env, synth.make_problem(17, 23, 3, [40, 64, 70], p=5, k=k, seed=960 + k, cap_frac=0.9), 0)


@pytest.mark.parametrize("m", [[1, 1], [15, 16], [17, 31], [33, 63], [65, 128], [129, 150]])
@pytest.mark.parametrize("mode", [0, 1])
def test_plain_sample_counts(env, m, mode):
    _check(env, synth.make_problem(16, 40, 2, m, p=3, k=18, seed=970 + m[0], cap_frac=0.9), mode)


@pytest.mark.parametrize("H,W", [(1, 127), (1, 128), (1, 129), (3, 85), (16, 16), (257, 1)])
def test_plain_pixel_counts(env, H, W):
    _check(env, synth.make_problem(H, W, 1, 9, p=3, k=40, seed=980 + W, cap_frac=0.9), 0)


@pytest.mark.parametrize("H,W", [(151, 129), (152, 257)])  # 77 x 4 and 153 x 4 units of 256 pixels
def test_plain_tile_rule(env, H, W):
    pr = synth.make_problem(H, W, 4, [70, 5, 64, 130], p=5, k=50, seed=990 + W)
    pix = np.unique(np.random.default_rng(1).integers(0, H * W, 3000)).astype(np.int32)
    _check(env, pr, 0, pix)


def test_plain_far_first_samples(env):
    """Samples ordered from far to near: the running maximum moves by thousands
    of log2 units between tiles and the last tile decides the sum."""
    pr = synth.make_problem(12, 400, 1, 500, p=3, k=18, seed=999, cap_frac=0.9)
    x = pr.sample_pix % 400
    pr.sample_pix = np.ascontiguousarray(pr.sample_pix[np.argsort(-np.abs(x - 3), kind="stable")])
    _check(env, pr, 0)
