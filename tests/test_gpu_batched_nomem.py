"""A batched call that fails for want of device memory leaves the context's work lists right for the calls after it."""
import numpy as np
import pytest

from gpu_util import to_dev
from paper_1908_06936_gb300 import synth

pytestmark = pytest.mark.gpu


# EXA_FP64 in one persistent launch, EXA_MIXED_FP32, EXA_MIXED_TF32X3, EXA_FP64 on the tensor cores
@pytest.mark.parametrize("prec,tile", [(0, 32), (1, 64), (3, 0), (0, 0)])
def test_a_failed_call_is_built_anew(prec, tile):
    import torch
    import paper_1908_06936_gb300 as exa

    def batch(sides):
        ns = [m * m for m in sides]
        locs = [to_dev(synth.jittered_grid(m, m)) for m in sides]
        return ns, locs, [to_dev(synth.normals(n, n)) for n in ns], to_dev(np.tile([1.0, 0.1, 0.5], len(ns)))

    def call(c, b):
        ns, locs, z, th = b
        out = torch.full((len(ns),), 7.0, dtype=torch.float64, device="cuda")
        st = torch.zeros(len(ns), dtype=torch.int32, device="cuda")
        rc = exa.exa_loglik_batched(c.handle, len(ns), ns, locs, z, th, prec, out, st)
        torch.cuda.synchronize()
        return rc, out.cpu().numpy(), st.cpu().numpy()

    small, large = batch([11, 20, 16]), batch([60, 48, 60, 55, 60, 60])
    with exa.Context() as c:
        c.check(exa.exa_ctx_set_batched(c.handle, tile, 0, 0, 0))
        ref = [call(c, b) for b in (small, large)]
    assert all(rc == 0 and np.all(st == 0) for rc, _, st in ref)
    with exa.Context() as c:
        c.check(exa.exa_ctx_set_batched(c.handle, tile, 0, 0, 0))
        assert call(c, small)[0] == 0
        free, _ = torch.cuda.mem_get_info()
        held = torch.empty(free - (200 << 20), dtype=torch.uint8, device="cuda")  # 200 MB left, the large batch takes 500
        assert call(c, large)[0] == exa.EXA_ERR_NOMEM
        rc, out, _ = call(c, small)
        assert rc == 0 and np.array_equal(out, ref[0][1])
        assert call(c, large)[0] == exa.EXA_ERR_NOMEM
        del held
        torch.cuda.empty_cache()
        for b, r in ((large, ref[1]), (small, ref[0])):
            rc, out, _ = call(c, b)
            assert rc == 0 and np.array_equal(out, r[1])
