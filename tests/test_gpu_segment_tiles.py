"""cs_segment over the shapes where its on-chip tiling can go wrong: one block,
ragged last tiles, one-pixel-wide images, several pixels per thread, label
counts around the kernels' instantiations (8 / 9, 16 / 17), with and without the
label cost whose sums cross all blocks. Bar as in test_gpu_segment.py: max
|u - u_ref| <= 2e-3 against the FP64 reference (non-expansive steps), labels
equal where the top two indicators differ by more than 1e-2.
"""
import numpy as np
import pytest

from oracle import segment as oseg

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


@pytest.mark.parametrize("nu", [0.0, 30.0])
@pytest.mark.parametrize("H,W,n,iters", [
    (5, 7, 3, 30),        # one block
    (1, 300, 2, 30), (300, 1, 4, 30), (2, 129, 16, 30),
    (61, 83, 8, 40), (61, 83, 9, 40), (47, 131, 16, 40), (47, 53, 17, 40),
    (97, 211, 1, 5),
    (331, 353, 5, 15),    # two pixels per thread
    (401, 521, 3, 10),    # four
    (321, 481, 16, 6),    # the windows fill the shared memory
    (480, 640, 12, 3),    # the state does not fit: global memory
])
def test_segment_tiles(env, H, W, n, iters, nu):
    cs, ctx, torch = env
    rng = np.random.default_rng(H * W + n)
    f = rng.uniform(0, 3, (n, H, W)).astype(np.float32)
    f -= 1.5 * (np.arange(n)[:, None, None] == (np.arange(W)[None, None, :] * n // W))
    img = rng.uniform(0, 1, (H, W, 3)).astype(np.float32)
    out = ctx.segment(_dev(torch, f), _dev(torch, img),
                      cs.SegParams.default(lam=5.0, nu=nu, iterations=iters))
    ctx.sync()
    u = out["u"].cpu().numpy().astype(np.float64)
    u_ref, lab_ref = oseg.segment(f.astype(np.float64), img, 5.0, nu=nu, iterations=iters)
    assert float(np.max(np.abs(u - u_ref))) <= 2e-3
    if n > 1:
        srt = np.sort(u_ref, axis=0)
        clear = (srt[-1] - srt[-2]) > 1e-2
        assert np.array_equal(out["labels"].cpu().numpy()[clear], lab_ref[clear])


def test_segment_back_to_back(env):
    """Launches that follow each other on one stream reuse the exchange planes
    and flags: every call gives the first one's bits."""
    cs, ctx, torch = env
    rng = np.random.default_rng(5)
    f = _dev(torch, rng.uniform(0, 3, (6, 90, 110)).astype(np.float32))
    img = _dev(torch, rng.uniform(0, 1, (90, 110, 3)).astype(np.float32))
    sp = cs.SegParams.default(lam=5.0, nu=20.0, iterations=25)
    outs = [ctx.segment(f, img, sp) for _ in range(6)]
    ctx.sync()
    for o in outs[1:]:
        assert torch.equal(o["u"], outs[0]["u"]) and torch.equal(o["labels"], outs[0]["labels"])
