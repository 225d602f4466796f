"""The give-up path of the bounded waits in the forms that test_gpu_timeout.py's
calls do not reach: the solver's tile form with a label cost (which also waits for
the blocks' sums) and its general form (grid barriers; more than 16 labels), the plain
FP32 sum's wait for its tensor-core products, and the tensor-core codes (pipelined,
and the kernel for operators too large for that). As there: the one-shot hook makes
one wait run out before anything is in flight, the call reports the timeout within
the shortened limit, and the next call gives the earlier bits.
"""
import re
import time

import numpy as np
import pytest

from paper_1312_4746_gb300 import synth

pytestmark = pytest.mark.gpu

LIMIT_NS = 20_000_000  # 20 ms: far above any normal wait of these launches


@pytest.fixture(scope="module")
def env(cuda_lib):
    import torch

    import paper_1312_4746_gb300 as cs

    ctx = cs.Context(0)
    yield cs, ctx, torch
    ctx.test_wait(0, cs.STALL_NONE)
    ctx.close()


def _stalled(cs, ctx, stall, call):
    """Runs `call` with the stall armed: the site of the wait that gave up."""
    ctx.test_wait(LIMIT_NS, stall)
    t0 = time.perf_counter()
    call()
    with pytest.raises(cs.CsError) as ei:
        ctx.sync()
    dt = time.perf_counter() - t0
    ctx.test_wait(0, cs.STALL_NONE)
    assert ei.value.status == cs.CS_ERR_TIMEOUT, ei.value
    assert dt < 0.5, dt  # the shortened limit, not the default 1 s
    return int(re.search(r"site (\d+)", str(ei.value)).group(1))


@pytest.mark.parametrize("n,nu", [(3, 0.0), (3, 30.0), (16, 30.0), (17, 0.0), (17, 30.0)])
def test_segment_forms(env, n, nu):
    cs, ctx, torch = env
    g = torch.Generator(device="cuda:0").manual_seed(n)
    f = 3.0 * torch.rand((n, 64, 96), generator=g, device="cuda:0")
    img = torch.rand((64, 96, 3), generator=g, device="cuda:0")
    sp = cs.SegParams.default(lam=2.0, nu=nu, iterations=20)
    ref = ctx.segment(f, img, sp)
    ctx.sync()
    assert _stalled(cs, ctx, cs.STALL_SEGMENT, lambda: ctx.segment(f, img, sp)) == 41
    out = ctx.segment(f, img, sp)
    ctx.sync()
    assert torch.equal(out["u"], ref["u"]) and torch.equal(out["labels"], ref["labels"])


@pytest.mark.parametrize("H,W,m", [(64, 96, [70, 5, 64, 130]),  # one operand tile per block
                                   (152, 257, [400, 5, 64, 430])])  # two
def test_plain_sum(env, H, W, m):
    cs, ctx, torch = env
    pr = synth.make_problem(H, W, 4, m, p=5, k=50, seed=77)
    img, om, mask, smp = (torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
                          for a in (pr.image, pr.omega, pr.mask, pr.sample_pix))
    prm = cs.Params.from_synth(pr.params)
    bits = ctx.codes(img, om, mask, prm)["bitmask"]

    def call(p=prm):
        return ctx.likelihood(img, bits, 50, pr.label_off, smp, p)["neglog"]

    ref = call()
    ctx.sync()
    assert _stalled(cs, ctx, cs.STALL_PLAIN, call) == 51
    assert torch.equal(call(), ref)
    # forms without that wait leave the stall armed
    ctx.test_wait(LIMIT_NS, cs.STALL_PLAIN)
    call(cs.Params.from_synth(pr.params, mode=cs.MODE_FACTORISED))
    call(cs.Params.from_synth(pr.params, precision=cs.FP8))
    ctx.sync()
    ctx.test_wait(0, cs.STALL_NONE)
    assert torch.equal(call(), ref)
    ctx.sync()


@pytest.mark.parametrize("p,k", [(5, 50), (9, 98), (9, 256)])
def test_codes(env, p, k):
    cs, ctx, torch = env
    pr = synth.make_problem(64, 96, 2, 20, p=p, k=k, seed=78)
    img, om, mask = (torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")
                     for a in (pr.image, pr.omega, pr.mask))
    prm = cs.Params.from_synth(pr.params, codes_form=cs.CODES_TC)

    def call(q=prm):
        return ctx.codes(img, om, mask, q)["bitmask"]

    ref = call()
    ctx.sync()
    # the first wait to give up records its site: the stalled one or one that
    # depends on it
    assert 20 <= _stalled(cs, ctx, cs.STALL_CODES, call) <= 27
    assert torch.equal(call(), ref)
    ctx.test_wait(LIMIT_NS, cs.STALL_CODES)  # a form without that wait leaves it armed
    assert torch.equal(call(cs.Params.from_synth(pr.params, codes_form=cs.CODES_FP32)), ref)
    ctx.sync()
    ctx.test_wait(0, cs.STALL_NONE)
    assert torch.equal(call(), ref)
    ctx.sync()
