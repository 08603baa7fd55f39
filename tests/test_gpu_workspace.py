"""Calls under a workspace bound: memory that a call does without is given back to the calls after it."""
import numpy as np
import pytest

from gpu_util import to_dev
from paper_1908_06936_gb300 import synth

pytestmark = pytest.mark.gpu

FP64, TF32X3 = 0, 3


def batch(sides):
    ns = [m * m for m in sides]
    return (ns, [to_dev(synth.jittered_grid(m, m)) for m in sides], [to_dev(synth.normals(n, n)) for n in ns],
            to_dev(np.tile([1.0, 0.1, 0.5], len(ns))))


def evaluate(c, b, prec):
    import torch
    import paper_1908_06936_gb300 as exa

    ns, locs, z, th = b
    out = torch.full((len(ns),), 7.0, dtype=torch.float64, device="cuda")
    st = torch.zeros(len(ns), dtype=torch.int32, device="cuda")
    c.check(exa.exa_loglik_batched(c.handle, len(ns), ns, locs, z, th, prec, out, st))
    torch.cuda.synchronize()
    assert np.all(st.cpu().numpy() == 0)
    return out.cpu().numpy()


def field(m):
    return to_dev(synth.jittered_grid(m, m)), to_dev(synth.normals(m * m, m))


def least(call):
    """The smallest bound (to 4 KB) under which a fresh context makes the call."""
    import paper_1908_06936_gb300 as exa

    def fits(bound):
        with exa.Context(workspace_bytes=bound) as c:
            try:
                call(c)
            except exa.ExaError as e:
                assert e.status == exa.EXA_ERR_NOMEM, e
                return False
            return True

    hi = 1 << 20
    while not fits(hi):
        hi *= 2
    lo = hi // 2
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if fits(mid) else (mid, hi)
    return hi


def test_fp64_batches_give_way_to_other_calls():
    # the mixed batch takes all that the FP64 batch on the tensor cores holds, and so does a single field
    import paper_1908_06936_gb300 as exa

    b = batch([30, 22, 35, 40])
    locs, z = field(48)
    theta = (1.0, 0.1, 0.5)
    calls = [lambda c: evaluate(c, b, TF32X3), lambda c: c.loglik(locs, z, theta)]
    for call in calls:
        bound = least(call)
        with exa.Context() as c:
            ref = call(c)
            first = evaluate(c, b, FP64)
        with exa.Context(workspace_bytes=bound + (32 << 20)) as c:  # room for the batch's 29 MB of matrices beside
            evaluate(c, b, FP64)
            held = exa.exa_workspace_bytes(c.handle)
        with exa.Context(workspace_bytes=max(bound, held)) as c:
            assert np.all(np.abs(evaluate(c, b, FP64) - first) <= 1e-10 * np.abs(first))
            got = call(c)
            assert np.all(np.abs(got - ref) <= 1e-10 * np.abs(ref))


def test_a_small_fp64_batch_gives_way_to_a_large_one():
    # the large batch has no room for the tensor-core form and runs in one persistent launch, alone in the bound
    import paper_1908_06936_gb300 as exa

    small, large = batch([30, 22, 35]), batch([40, 48, 44])
    bound = least(lambda c: evaluate(c, large, FP64))
    with exa.Context() as c:
        ref = evaluate(c, large, FP64)
    with exa.Context(workspace_bytes=bound) as c:
        evaluate(c, small, FP64)
        assert np.all(np.abs(evaluate(c, large, FP64) - ref) <= 1e-10 * np.abs(ref))


def test_every_kind_of_spare_memory_is_given_back():
    # a mixed batch's second panel operand, an FP64 batch and an FP64 evaluation's digits are held together; the last
    # call needs the room of all three
    import paper_1908_06936_gb300 as exa

    b = batch([30, 22, 35])
    small, large = field(30), field(60)
    theta = (1.0, 0.1, 0.5)

    def before(c):
        evaluate(c, b, TF32X3)
        evaluate(c, b, FP64)
        c.loglik(*small, theta)

    with exa.Context(tile_nb=64) as c:  # tile 64 takes no digits, and a CTA count no tensor-core batch
        evaluate(c, b, TF32X3)
        with_spare = exa.exa_workspace_bytes(c.handle)
    with exa.Context(workspace_bytes=with_spare - 1) as c:
        evaluate(c, b, TF32X3)
        batch_bytes = exa.exa_workspace_bytes(c.handle)  # without the second panel operand
    bound = batch_bytes + least(lambda c: c.loglik(*large, theta))
    with exa.Context() as c:
        before(c)
        assert exa.exa_workspace_bytes(c.handle) < bound
        ref = c.loglik(*large, theta)
    with exa.Context(workspace_bytes=bound) as c:
        before(c)
        assert abs(c.loglik(*large, theta) - ref) <= 1e-10 * abs(ref)
