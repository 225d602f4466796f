"""A kernel's limit of dynamic shared memory belongs to the device, not to a context:
two threads with a context each, whose calls need different amounts in the same
kernel (the k-medians histograms, 8 KB a class), must not disturb one another
between setting the limit and the rounds' launches. Centres equal those of the same
call alone.
"""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_two_contexts_different_class_counts(cuda_lib):
    import torch

    import paper_1312_4746_gb300 as cs

    g = torch.Generator(device="cuda:0").manual_seed(11)
    V = torch.exp(-(0.14 * torch.randn((6, 3000), generator=g, device="cuda:0")) ** 2 / 0.01)
    V = V.contiguous()
    torch.cuda.synchronize()
    starts = {n: np.arange(n, dtype=np.int32) * 180 for n in (4, 16)}
    # 16 classes in few calls of many rounds (a long way from the limit's setting to
    # the last launch), 4 classes in many calls of none or one
    plan = {16: (300, 6), 4: (1, 1500)}
    want, errors = {}, []
    ctx = cs.Context(0)
    for n, (rounds, _) in plan.items():
        want[n] = ctx.kmedians(V, starts[n], rounds)["centres"].clone()
    ctx.sync()
    ctx.close()

    def work(n):
        try:
            c = cs.Context(0)
            s = torch.cuda.Stream()
            rounds, calls = plan[n]
            with torch.cuda.stream(s):
                for _ in range(calls):
                    out = c.kmedians(V, starts[n], rounds)
                c.sync()
            assert torch.equal(out["centres"], want[n])
            c.close()
        except Exception as e:  # reported by the main thread
            errors.append((n, repr(e)))

    threads = [threading.Thread(target=work, args=(n,)) for n in plan]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
