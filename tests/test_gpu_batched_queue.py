"""Batched calls that queue up behind other work on their stream, and captured ones that are replayed after other calls:
each keeps the locations and observations it was given."""
import numpy as np
import pytest

from gpu_util import to_dev
from paper_1908_06936_gb300 import synth

pytestmark = pytest.mark.gpu

SIDES = [9, 14, 20]
# EXA_FP64 on the tensor cores, EXA_FP64 in one persistent launch, EXA_MIXED_FP32, EXA_MIXED_TF32X3
FORMS = [(0, 0), (0, 32), (1, 64), (3, 0)]


class Batch:
    def __init__(self, seed, sides=SIDES):
        import torch

        self.ns = [m * m for m in sides]
        self.locs = [to_dev(synth.jittered_grid(m, seed + m)) for m in sides]
        self.z = [to_dev(synth.normals(m * m, seed + m)) for m in sides]
        self.theta = to_dev(np.tile([1.0, 0.1, 0.5], len(sides)))
        self.out = torch.zeros(len(sides), dtype=torch.float64, device="cuda")
        self.status = torch.zeros(len(sides), dtype=torch.int32, device="cuda")

    def call(self, c, prec):
        import paper_1908_06936_gb300 as exa

        c.check(exa.exa_loglik_batched(c.handle, len(self.ns), self.ns, self.locs, self.z, self.theta, prec, self.out,
                                       self.status))

    def take(self):
        got = self.out.cpu().numpy().copy()
        assert np.all(self.status.cpu().numpy() == 0)
        self.out.zero_()
        return got


@pytest.mark.parametrize("prec,tile", FORMS)
def test_queued_calls_keep_their_inputs(prec, tile):
    import torch
    import paper_1908_06936_gb300 as exa

    batches = [Batch(100 * k) for k in range(7)]
    with exa.Context() as c:
        c.check(exa.exa_ctx_set_batched(c.handle, tile, 0, 0, 0))
        ref = []
        for b in batches:
            b.call(c, prec)
            torch.cuda.synchronize()
            ref.append(b.take())
        torch.cuda._sleep(200_000_000)  # about 0.1 s, so that the calls below are enqueued before the first one runs
        for b in batches:
            b.call(c, prec)
        torch.cuda.synchronize()
        for b, r in zip(batches, ref):
            assert np.array_equal(b.take(), r)


@pytest.mark.parametrize("prec,tile", FORMS)
def test_a_replayed_graph_keeps_its_inputs(prec, tile):
    import torch
    import paper_1908_06936_gb300 as exa

    a, b = Batch(0), Batch(1000)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s), exa.Context(stream=s) as c:
        c.check(exa.exa_ctx_set_batched(c.handle, tile, 0, 0, 0))
        a.call(c, prec)
        s.synchronize()
        ref_a = a.take()
        b.call(c, prec)
        s.synchronize()
        ref_b = b.take()
        graphs = []
        for x in (a, b, a):
            graphs.append(torch.cuda.CUDAGraph())
            with torch.cuda.graph(graphs[-1], stream=s):
                x.call(c, prec)
        for k in range(2):  # replays, and a call with other inputs in between
            for g, x, ref in zip(graphs, (a, b, a), (ref_a, ref_b, ref_a)):
                g.replay()
                s.synchronize()
                assert np.array_equal(x.take(), ref)
            b.call(c, prec)
            s.synchronize()
            assert np.array_equal(b.take(), ref_b)


@pytest.mark.parametrize("prec,tile", FORMS)
def test_lists_built_under_capture_are_not_taken_for_built(prec, tile):
    # the first call of a smaller batch is captured (its buffers are there): its lists are on the device only while its
    # replay is the last call
    import torch
    import paper_1908_06936_gb300 as exa

    big, small = Batch(0), Batch(50, SIDES[:2])
    s = torch.cuda.Stream()

    def check(run, b, ref):
        run()
        s.synchronize()
        assert np.array_equal(b.take(), ref)

    with torch.cuda.stream(s), exa.Context(stream=s) as c:
        c.check(exa.exa_ctx_set_batched(c.handle, tile, 0, 0, 0))
        big.call(c, prec)
        s.synchronize()
        ref_big = big.take()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            small.call(c, prec)
        small.call(c, prec)
        s.synchronize()
        ref = small.take()
        with exa.Context(stream=s) as other:
            other.check(exa.exa_ctx_set_batched(other.handle, tile, 0, 0, 0))
            check(lambda: small.call(other, prec), small, ref)
        for _ in range(2):
            check(g.replay, small, ref)
            check(lambda: big.call(c, prec), big, ref_big)
            check(lambda: big.call(c, prec), big, ref_big)


def test_more_panels_than_a_grid_has_rows():
    # 33,000 fields with a panel: the splits of W and of L, one piece each a field, exceed the 65,535 of a grid's y dimension
    import torch
    import paper_1908_06936_gb300 as exa

    nrep, n = 33000, 129
    locs = [to_dev(synth.jittered_grid(12, s)[:n]) for s in range(3)]
    z = [to_dev(synth.normals(n, s)) for s in range(3)]
    theta = to_dev(np.tile([1.0, 0.1, 0.5], nrep))
    out = torch.zeros(nrep, dtype=torch.float64, device="cuda")
    status = torch.zeros(nrep, dtype=torch.int32, device="cuda")
    pick = [r % 3 for r in range(nrep)]
    with exa.Context() as c:
        ref = np.array([c.loglik(l, y, (1.0, 0.1, 0.5)) for l, y in zip(locs, z)])
        c.check(exa.exa_loglik_batched(c.handle, nrep, [n] * nrep, [locs[k] for k in pick], [z[k] for k in pick], theta,
                                       exa.EXA_FP64, out, status))
        torch.cuda.synchronize()
    assert np.all(status.cpu().numpy() == 0)
    got = out.cpu().numpy()
    assert np.all(np.abs(got - ref[pick]) <= 1e-10 * np.abs(ref[pick]))
