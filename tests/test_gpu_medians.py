"""Order statistics behind the texture classes and representatives, at the
sizes and values where their selection can go wrong.

cs_kmedians: after one round the centres are exactly the elementwise medians
of the members of the start assignment (FP32 mean of the two middle values for
an even count, order of the float bits: -0 below +0, NaN beyond the infinity of
its sign), so they are compared bit for bit with a sort on the host.
Majority co-supports (factorised form): a wrong bit moves L by several 1e-2
nats, the bar is the plain form's 1e-5 relative.
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


def _key(v):
    u = np.ascontiguousarray(v, np.float32).view(np.uint32)
    return np.where(u >> 31, ~u, u | np.uint32(0x80000000)).astype(np.uint32)


def _median(v):
    s = v[np.argsort(_key(v), kind="stable")]
    m = len(s)
    if m % 2:
        return s[m // 2]
    with np.errstate(invalid="ignore", over="ignore"):
        return np.float32(0.5) * (s[m // 2 - 1] + s[m // 2])


def _values(kind, rng, k, N):
    if kind == "iota":  # crowded near 0 and 1
        return np.exp(-rng.normal(0, 0.14, (k, N)) ** 2 / 0.01).astype(np.float32)
    if kind == "tiny":  # below every fine step of the first pass, denormals among them
        return (rng.uniform(0, 1, (k, N)) * 10.0 ** rng.uniform(-44, -12, (k, N))).astype(np.float32)
    if kind == "equal":  # one key: more than any list holds
        return np.full((k, N), 0.25, np.float32)
    if kind == "two":
        return rng.choice(np.array([0.5, 1.0], np.float32), (k, N))
    if kind == "wide":  # both signs, large, infinities
        v = (rng.normal(0, 1, (k, N)) * 10.0 ** rng.uniform(-6, 30, (k, N))).astype(np.float32)
        v[rng.random((k, N)) < 0.02] = np.inf
        return v
    edges = np.array([0.0, -0.0, 0.125, np.nextafter(np.float32(0.125), np.float32(0)), 1.0,
                      np.nextafter(np.float32(1), np.float32(0)),
                      np.nextafter(np.float32(1), np.float32(2)), 2.0 ** -35, 127 / 1024,
                      129 / 1024], np.float32)
    return rng.choice(edges, (k, N))


@pytest.mark.parametrize("kind", ["iota", "tiny", "equal", "two", "wide", "edges"])
@pytest.mark.parametrize("k,N,n", [(3, 1, 1), (5, 2, 2), (4, 5, 3), (3, 16385, 2), (2, 40003, 1),
                                   (7, 9000, 16), (6, 33000, 9)])
def test_kmedians_centres_exact(env, kind, k, N, n):
    cs, ctx, torch = env
    rng = np.random.default_rng(900 + N + n)
    V = _values(kind, rng, k, N)
    init = rng.choice(N, n, replace=False).astype(np.int32)
    Vd = _dev(torch, V)
    lab = ctx.kmedians(Vd, init, 0)["assign"].cpu().numpy()
    C = ctx.kmedians(Vd, init, 1)["centres"].cpu().numpy()
    ctx.sync()
    for b in range(n):
        mem = V[:, lab == b]
        want = np.array([_median(mem[j]) if mem.shape[1] else V[j, init[b]] for j in range(k)],
                        np.float32)
        np.testing.assert_array_equal(C[b], want)


def test_kmedians_nan_order(env):
    """A NaN sorts beyond the infinity of its sign; its point has no finite
    distance and goes to class 0."""
    cs, ctx, torch = env
    V = np.random.default_rng(7).uniform(0, 1, (3, 401)).astype(np.float32)
    V[0, 5] = np.nan
    V[1, 9] = -np.nan
    C = ctx.kmedians(_dev(torch, V), [0], 1)["centres"].cpu().numpy()
    ctx.sync()
    np.testing.assert_array_equal(C[0], [_median(V[j]) for j in range(3)])


@pytest.mark.parametrize("nl,m,p,k", [(3, [1, 31, 33], 5, 33), (2, [257, 32], 7, 98),
                                      (4, [2, 64, 255, 300], 3, 18)])
def test_majority_cosupport(env, nl, m, p, k):
    cs, ctx, torch = env
    pr = synth.make_problem(48, 61, nl, m, p=p, k=k, seed=910 + nl, cap_frac=0.9)
    pr.params.mode = 1
    prm = cs.Params.from_synth(pr.params)
    out = ctx.data_term(_dev(torch, pr.image), _dev(torch, pr.omega), _dev(torch, pr.mask),
                        pr.label_off, _dev(torch, pr.sample_pix), prm)
    ctx.sync()
    L = -out["neglog"].cpu().numpy().reshape(nl, -1).astype(np.float64)
    ref = oracle.data_term(pr)["L"]
    assert np.max(np.abs(L - ref) / np.maximum(np.abs(ref), 1.0)) <= 1e-5


@pytest.mark.parametrize("nl", [4, 9, 18])
def test_smooth_label_groups(env, nl):
    """More labels than one sweep's register sums hold: labels repeated from a
    three-label problem have equal likelihoods, and the posteriors are the
    three-label ones shared out."""
    cs, ctx, torch = env
    pr = synth.make_problem(33, 45, 3, 20, p=5, k=50, seed=930)
    prm = cs.Params.from_synth(pr.params, mode=cs.MODE_SMOOTH)
    img, om, mk = _dev(torch, pr.image), _dev(torch, pr.omega), _dev(torch, pr.mask)
    off = pr.label_off
    which = [i % 3 for i in range(nl)]
    pix = np.concatenate([pr.sample_pix[off[i]:off[i + 1]] for i in which])
    off2 = np.concatenate([[0], np.cumsum([off[i + 1] - off[i] for i in which])]).astype(np.int32)
    a = ctx.data_term(img, om, mk, off, _dev(torch, pr.sample_pix), prm)["post"].cpu().numpy()
    b = ctx.data_term(img, om, mk, off2, _dev(torch, pix), prm)["post"].cpu().numpy()
    ctx.sync()
    w = np.array([which.count(i) for i in range(3)], np.float64)
    # equal labels share the texture and the label softmax alike: p_i w_i under
    # a common factor, within the FP32 softmaxes' rounding
    e = a.astype(np.float64)
    e = e / (w[:, None, None] * e).sum(0)
    for i in range(nl):
        np.testing.assert_allclose(b[i], e[which[i]], rtol=3e-5, atol=1e-7)
