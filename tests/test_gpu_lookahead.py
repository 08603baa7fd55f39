"""Look-ahead shares of the mixed factorisation: however many SMs factor a diagonal block, every entry sees the same
operations in the same order, so the factor keeps its bits."""
import pytest

from gpu_util import to_dev
from paper_1908_06936_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beta", [0.05, 0.1])
def test_the_share_leaves_the_log_determinant_alone(beta):
    import paper_1908_06936_gb300 as exa

    m = 45  # four panels: the look-ahead stream factors the last three
    locs, z = to_dev(synth.jittered_grid(m, m)), to_dev(synth.normals(m * m, m))
    theta = (1.0, beta, 0.5)
    with exa.Context() as c:
        ref = c.loglik_ex(locs, z, theta, exa.EXA_MIXED_TF32X3)
    for share in (1, 2, 3, 4, 5, 6, 7, 8, 9, 20, 33):
        with exa.Context() as c:
            c.check(exa.exa_ctx_set_lookahead(c.handle, share))
            c.check(exa.exa_ctx_set_lookahead_late(c.handle, 0, 0))  # the share as it is, at every size
            got = c.loglik_ex(locs, z, theta, exa.EXA_MIXED_TF32X3)
        assert got["logdet"] == ref["logdet"], share
