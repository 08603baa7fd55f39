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


def padded(n):
    return -(-n // 128) * 128


def fp64_units_bytes(n):
    """What the FP64 evaluation on the FP64 units holds: the matrix, the tile inverses, the panel, log-determinant parts,
    three vectors, the reductions' partial sums and the interpolation table."""
    import paper_1908_06936_gb300 as exa

    npad = padded(n)
    with exa.Context() as c:
        c.covariance(to_dev(synth.uniform_square(4, 1)), (1.0, 0.1, 0.5))
        table = exa.exa_workspace_bytes(c.handle)
    return 8 * (npad * npad + 2 * npad * 128 + npad // 128 + 3 * npad + 1024 + (npad // 1024 + 2) * 128) + table


@pytest.mark.parametrize("n", [100, 700, 1300])
def test_the_fp64_evaluation_needs_no_more_than_the_fp64_units(n):
    import paper_1908_06936_gb300 as exa

    locs, z = to_dev(synth.jittered_grid(37, n)[:n]), to_dev(synth.normals(n, n))
    theta = (1.0, 0.1, 0.5)
    with exa.Context() as c:
        ref = c.loglik(locs, z, theta)
    with exa.Context(workspace_bytes=fp64_units_bytes(n)) as c:
        assert abs(c.loglik(locs, z, theta) - ref) <= 1e-10 * abs(ref)


@pytest.mark.parametrize("n,m,extra", [(1300, 600, 0), (1300, 600, 4 << 20), (1300, 600, 12 << 20), (1300, 600, 24 << 20),
                                       (700, 2048, 0), (700, 2048, 6 << 20), (700, 2048, 16 << 20)])
def test_a_prediction_needs_no_more_than_the_fp64_units(n, m, extra):
    # beside the evaluation: 512 columns of cross covariances and of a 128-row solve, and their sums; more room leaves
    # some of the digit operands in, but not all
    import paper_1908_06936_gb300 as exa

    locs, z = to_dev(synth.jittered_grid(37, n)[:n]), to_dev(synth.normals(n, n))
    new, theta = to_dev(synth.uniform_square(m, m + 1)), (1.0, 0.1, 0.5)
    with exa.Context() as c:
        ref = [t.cpu().numpy() for t in c.predict(locs, z, theta, new)]
    bound = fp64_units_bytes(n) + 8 * 512 * (padded(n) + 129) + extra
    with exa.Context(workspace_bytes=bound) as c:
        got = [t.cpu().numpy() for t in c.predict(locs, z, theta, new)]
        again = [t.cpu().numpy() for t in c.predict(locs, z, theta, new)]
        assert exa.exa_workspace_bytes(c.handle) <= bound
    for g, a, r, scale in zip(got, again, ref, (float(z.abs().max()), theta[0])):
        assert np.all(np.abs(g - r) <= 1e-9 * scale) and np.all(np.abs(a - r) <= 1e-9 * scale)


def test_fisher_needs_no_more_than_the_fp64_units():
    # five padded matrices, the partial sums, the tile inverses, the panel, log-determinant parts and the table
    import paper_1908_06936_gb300 as exa

    n = 700
    npad, locs, theta = padded(n), to_dev(synth.jittered_grid(27, 3)[:n]), (1.0, 0.1, 0.5)
    with exa.Context() as c:
        ref = c.fisher(locs, theta)
    units = fp64_units_bytes(n) - 8 * (3 * npad + 1024 + (npad // 1024 + 2) * 128)
    for extra in (0, 4 << 20, 9 << 20):
        with exa.Context(workspace_bytes=units + 8 * (4 * npad * npad + (npad // 32) ** 2 * 6) + extra) as c:
            assert np.all(np.abs(c.fisher(locs, theta) - ref) <= 1e-9 * np.abs(ref))


def test_a_prediction_gives_way_to_a_larger_field():
    # the prediction's blocks of 2,048 points go when the field needs their room; those of 512 points stay
    import paper_1908_06936_gb300 as exa

    n, large = 900, 2200
    locs, z = to_dev(synth.jittered_grid(30, 1)), to_dev(synth.normals(n, 1))
    new, theta = to_dev(synth.uniform_square(2048, 5)), (1.0, 0.1, 0.5)
    big, zbig = to_dev(synth.jittered_grid(47, 2)[:large]), to_dev(synth.normals(large, 2))
    with exa.Context() as c:
        ref = c.loglik(big, zbig, theta)
    with exa.Context(workspace_bytes=fp64_units_bytes(large) + 8 * 512 * (padded(n) + 129)) as c:
        c.predict(locs, z, theta, new)
        assert abs(c.loglik(big, zbig, theta) - ref) <= 1e-10 * abs(ref)


# Calls on one context, and the bytes they left held when the FP64 calls ran on the FP64 units and the mixed ones without
# the 512-wide block inverses.  ll, g, f, p, s: log-likelihood, gradient, Fisher information, prediction of 2,500 points,
# simulation of n points in FP64; mx, gm, sm: the mixed ones; b32: FP64 batch in one launch, bt: mixed batch.
SEQUENCES = [
    ("ll1024 mx1500", 77165456),
    ("ll1024 gm1024", 75418664),
    ("ll1024 sm1500", 57900432),
    ("mx1024 mx1500", 76747664),
    ("mx1024 sm1500", 66065296),
    ("g513 gm2100", 256875640),
    ("f513 mx1500", 89874064),
    ("mx513 gm400 btL b32S", 174693936),
    ("p513 f100 gm513 s513", 78688160),
    ("f513 gm400 s1024 s1024", 57964128),
    ("mx400 p513 mx513 f2100", 232764080),
    ("s100 g400 gm1024 sm513", 77110312),
    ("p100 sm1024 mx513 ll1500", 58631048),
]
SMALL, LARGE = [20, 11, 26], [30, 41, 22, 36]


def make(name):
    import paper_1908_06936_gb300 as exa

    theta = (1.0, 0.1, 0.5)
    kind, size = name.rstrip("0123456789SL"), name.lstrip("bcdefghijklmnopqrstuvwxyz")
    if name.startswith("b"):
        def call(c):
            c.check(exa.exa_ctx_set_batched(c.handle, 32 if name.startswith("b32") else 0, 0, 0, 0))
            return evaluate(c, batch(SMALL if name.endswith("S") else LARGE), FP64 if name.startswith("b32") else TF32X3)
        return call
    n = int(size)
    locs, z = to_dev(synth.jittered_grid(int(np.ceil(n ** 0.5)), n)[:n]), to_dev(synth.normals(n, n))
    return {
        "ll": lambda c: c.loglik(locs, z, theta),
        "mx": lambda c: c.loglik(locs, z, theta, TF32X3),
        "g": lambda c: c.loglik_grad(locs, z, theta)[1],
        "gm": lambda c: c.loglik_grad(locs, z, theta, TF32X3)[1],
        "f": lambda c: c.fisher(locs, theta),
        "p": lambda c: c.predict(locs, z, theta, to_dev(synth.uniform_square(2500, 9)))[0].cpu().numpy(),
        "s": lambda c: c.simulate(locs, z, theta).cpu().numpy(),
        "sm": lambda c: c.simulate(locs, z, theta, TF32X3).cpu().numpy(),
    }[kind]


@pytest.mark.parametrize("calls,bound", SEQUENCES)
def test_a_sequence_needs_no_more_than_without_the_spare_memory(calls, bound):
    # the results are those of each call on a context of its own: to 1e-8 of the largest, the bar of the quadratic forms
    import paper_1908_06936_gb300 as exa

    with exa.Context(workspace_bytes=bound) as c:
        for name in calls.split():
            call = make(name)
            got = np.asarray(call(c))
            with exa.Context() as fresh:
                ref = np.asarray(call(fresh))
            assert np.all(np.abs(got - ref) <= 2e-8 * np.max(np.abs(ref))), name
        assert exa.exa_workspace_bytes(c.handle) <= bound
