"""How accurate the FP64 paths are, beyond agreeing with the oracle: rounding errors that a step must not add."""
import numpy as np
import pytest

from gpu_util import to_dev
from paper_1908_06936_gb300 import synth

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("seed", range(4))
def test_diagonal_block_rounds_once_a_step(seed):
    # A diagonal entry of the last 128 rows is rounded once for each of at most 16 steps of 32 columns and by up to 32
    # columns of its own leaf, each time by at most u A_ii: with independent errors of a third of that in the mean square,
    # sqrt(48 / 3) u A_ii = 4 u A_ii.  Rounded at each of the up to 512 columns it came to 6 to 7.
    import torch
    import paper_1908_06936_gb300 as exa

    n = 512
    rng = np.random.default_rng(seed)
    g = rng.standard_normal((n, n // 2)) / np.sqrt(n // 2)
    a = g @ g.T + np.eye(n)
    a = 0.5 * (a + a.T)
    buf = torch.as_tensor(a, device="cuda")
    with exa.Context() as c:
        c.check(exa.exa_potrf(c.handle, buf, n, n))
    l = np.triu(buf.cpu().numpy()).T.astype(np.longdouble)
    resid = ((l * l).sum(1) - np.diag(a))[384:] / np.diag(a)[384:]
    assert np.sqrt(np.mean(resid.astype(float) ** 2)) <= 4 * U
