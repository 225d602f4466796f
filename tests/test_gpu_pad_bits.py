"""The texture similarity is over the k codes: whatever a caller's bitmasks hold in
the last word's bits beyond them changes nothing, in every form that takes bitmasks
(likelihood, batch with given codes, surrogate). Bit for bit the result of clean
bitmasks. k + 2 columns of the plain form's operand share the codes' words (k = 50)
or not (k = 31), some tensor-core texture codes ride in another slab (k = 98), or no
bit is left over (k = 64).
"""
import numpy as np
import pytest

from paper_1312_4746_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(cuda_lib):
    import torch

    import paper_1312_4746_gb300 as cs

    ctx = cs.Context(0)
    yield cs, ctx, torch
    ctx.close()


def _problem(env, k):
    cs, ctx, torch = env
    pr = synth.make_problem(40, 61, 3, [20, 64, 90], p=7, k=k, seed=700 + k)
    img, om, mask, smp = (torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
                          for a in (pr.image, pr.omega, pr.mask, pr.sample_pix))
    out = ctx.codes(img, om, mask, cs.Params.from_synth(pr.params), want_lead16=True)
    clean = out["bitmask"]
    dirty = clean.clone()
    if k % 32:
        pad = np.random.default_rng(k).integers(0, 2 ** 32, len(clean), np.uint64)
        pad &= np.uint64((0xFFFFFFFF << (k % 32)) & 0xFFFFFFFF)
        dirty[:, -1] |= torch.from_numpy(pad.astype(np.uint32).view(np.int32)).to("cuda:0")
    return pr, img, smp, clean, dirty, out["lead16"]


@pytest.mark.parametrize("k", [31, 50, 64, 98])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("precision,l_tol", [(0, 1e-3), (1, 1e-3), (2, 1e-3), (2, 1e-9)])
def test_likelihood(env, k, mode, precision, l_tol):
    cs, ctx, torch = env
    pr, img, smp, clean, dirty, _ = _problem(env, k)
    prm = cs.Params.from_synth(pr.params, mode=mode, precision=precision, l_tol=l_tol)
    a = ctx.likelihood(img, clean, k, pr.label_off, smp, prm)
    b = ctx.likelihood(img, dirty, k, pr.label_off, smp, prm)
    images = [{"img": img, "sample_pix": smp, "label_off": pr.label_off, "bitmask": dirty}]
    c = ctx.batch_likelihood(images, k, prm)[0]
    ctx.sync()
    for out in (b, c):
        assert torch.equal(out["neglog"], a["neglog"]) and torch.equal(out["post"], a["post"])


@pytest.mark.parametrize("mode", [0, 1])
def test_surrogate(env, mode):
    cs, ctx, torch = env
    k = 50
    pr, img, smp, clean, dirty, lead = _problem(env, k)
    prm = cs.Params.from_synth(pr.params, mode=mode)
    got = []
    for bits in (clean, dirty):
        args = (img, bits, lead, k, pr.label_off, smp, prm)
        ctx.surrogate_fit(*args, frac=0.2, steps=5)
        got.append(ctx.surrogate_eval(*args, margin=0.3, rule=cs.FALLBACK_MARGIN))
    ctx.sync()
    assert got[0][1] == got[1][1]
    assert torch.equal(got[0][0]["neglog"], got[1][0]["neglog"])
