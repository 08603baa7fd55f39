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


@pytest.mark.parametrize("nu,beta,bound", [(2.5, 0.2, 1.2e-7), (3.5, 0.15, 3e-5)])
def test_log_determinant_of_smooth_fields(nu, beta, bound):
    # 1,024 points, against the FP64 units (tile 64).  In 80-bit arithmetic 128-wide panels on the FP64 units leave
    # errors of 3.1e-8 and 5.4e-6 (root mean square of 16 fields), panels with a correction from two digits 3.4e-7 and
    # 2.0e-3, from four 7e-9 and 8e-7.  Bound: four times the FP64 units' own, and a margin for four fields.
    import paper_1908_06936_gb300 as exa

    diff = []
    for seed in range(1, 5):
        locs, z = to_dev(synth.jittered_grid(32, seed)), to_dev(synth.normals(1024, seed))
        with exa.Context(tile_nb=128) as c, exa.Context(tile_nb=64) as units:
            diff.append(c.loglik_ex(locs, z, (1.0, beta, nu))["logdet"] - units.loglik_ex(locs, z, (1.0, beta, nu))["logdet"])
    assert np.sqrt(np.mean(np.square(diff))) <= bound, diff


@pytest.mark.parametrize("nu,beta,bound", [(0.5, 0.1, 2.5e-15), (1.0, 0.05, 2.5e-15), (2.5, 0.1, 3e-14), (2.5, 0.2, 1e-13)])
def test_kriging_variance_against_the_fp64_units(nu, beta, bound):
    # 1,024 points, the largest difference from tile 64 (the FP64 units).  In 80-bit arithmetic with one and the same
    # factor, 128-wide inverses on the FP64 units leave 9.3e-16, 1.2e-15, 1.1e-14 and 2.2e-14, 512-wide ones as digit
    # products 4.0e-15, 4.2e-15, 2.7e-13 and 1.1e-12, and once corrected 6e-16, 8e-16, 5e-16 and 1e-15.  Bound: the FP64
    # units' error and a margin for the maximum over three fields and for the two factors.
    import paper_1908_06936_gb300 as exa

    diff = []
    for seed in range(1, 4):
        locs, z = to_dev(synth.jittered_grid(32, seed)), to_dev(synth.normals(1024, seed))
        new = to_dev(synth.uniform_square(256, seed + 50))
        with exa.Context(tile_nb=128) as c, exa.Context(tile_nb=64) as units:
            a, b = (x.predict(locs, z, (1.0, beta, nu), new)[1].cpu().numpy() for x in (c, units))
        diff.append(np.max(np.abs(a - b)))
    assert max(diff) <= bound, diff


@pytest.mark.parametrize("nu,beta,bound", [(2.5, 0.2, 4e-10), (3.5, 0.15, 2.5e-8)])
def test_batched_log_likelihood_of_smooth_fields(nu, beta, bound):
    # eight fields of 529 points, relative difference from the persistent form (root mean square).  In 80-bit arithmetic
    # the persistent form's 64-wide tiles leave 1.3e-10 and 5.5e-9 (16 fields), 128-wide inverses as digit products
    # 6.8e-10 and 8.2e-8, and once corrected 3.6e-11 and 1.4e-9.  Bound: the persistent form's error, and a factor of 3
    # to 4.5 for the smaller sample.
    import torch
    import paper_1908_06936_gb300 as exa

    locs = [to_dev(synth.jittered_grid(23, seed)) for seed in range(1, 9)]
    z = [to_dev(synth.normals(529, seed)) for seed in range(1, 9)]
    theta = to_dev(np.tile([1.0, beta, nu], 8))
    got = []
    with exa.Context() as c:
        for ctas in (0, 1):
            out = torch.empty(8, dtype=torch.float64, device="cuda")
            st = torch.empty(8, dtype=torch.int32, device="cuda")
            c.check(exa.exa_ctx_set_batched(c.handle, 64, ctas, 0, 0))
            c.check(exa.exa_loglik_batched(c.handle, 8, [529] * 8, locs, z, theta, exa.EXA_FP64, out, st))
            torch.cuda.synchronize()
            assert np.all(st.cpu().numpy() == 0)
            got.append(out.cpu().numpy())
    rel = (got[0] - got[1]) / got[1]
    assert np.sqrt(np.mean(rel ** 2)) <= bound, rel


@pytest.mark.parametrize("x", [20.0, 31.0, 40.0, 63.0, 64.5, 70.0, 90.0, 91.0, 120.0, 150.0])
def test_range_derivative_of_far_points(x):
    # A 21 x 22 grid with spacing x beta, nu = 1/2: Sigma = sigma^2 (I + E) with E of size exp(-x), so its inverse is
    # (I - E) / sigma^2 to exp(-2 x), and dl/dbeta = 1/2 sum_ij (a_i a_j - S_ij) D_ij, D = sigma^2 (r / beta^2) exp(-r / beta),
    # is carried by the pairs at distance x and a few more.  An entry is off by the rounding of r^2 / beta^2 (2 u
    # relative, x u in the exponential), of the piece's coordinate (no more) and of the polynomial: 4 x u of the sum of the
    # absolute values bounds it with room for the sum.
    import paper_1908_06936_gb300 as exa

    sigma2, beta = 1.3, 0.01
    i, j = np.meshgrid(np.arange(21), np.arange(22), indexing="ij")
    locs = np.stack([i.ravel(), j.ravel()], 1) * (x * beta)
    z = synth.normals(len(locs), 7)
    with exa.Context() as c:
        g = c.loglik_grad(to_dev(locs), to_dev(z), (sigma2, beta, 0.5))[1]
    r = np.sqrt(((locs[:, None].astype(np.longdouble) - locs[None]) ** 2).sum(-1))
    e = np.exp(-r / np.longdouble(beta))
    d = sigma2 * r / np.longdouble(beta) ** 2 * e
    e[np.diag_indices(len(e))] = 0
    ez = (e * z[None]).sum(1)
    a = (z - ez + (e * ez[None]).sum(1)) / sigma2
    terms = 0.5 * (a[:, None] * a[None] + e / sigma2) * d  # D is zero on the diagonal
    assert abs(float(g[1] - terms.sum())) <= 4 * x * U * float(np.abs(terms).sum())


@pytest.mark.parametrize("m,nu,beta", [(20, 3.5, 1.0), (32, 3.0, 1.0), (32, 3.5, 0.3), (32, 4.5, 0.2), (45, 3.0, 0.5), (45, 3.5, 0.3)])
def test_smooth_fields_that_the_fp64_units_factor(m, nu, beta):
    # close to the limit of FP64, a lost digit shows as a failed pivot: what the FP64 units (tile 64, persistent batch)
    # factor, the digit products factor too
    import torch
    import paper_1908_06936_gb300 as exa

    theta = (1.0, beta, nu)
    for seed in (1, 2):
        locs, z = to_dev(synth.jittered_grid(m, seed)), to_dev(synth.normals(m * m, seed))
        with exa.Context(tile_nb=64) as units:
            ok = exa.exa_loglik_ex(units.handle, locs, z, theta, m * m, exa.EXA_FP64, exa.ExaResult()) == exa.EXA_OK
        with exa.Context() as c:
            st = exa.exa_loglik_ex(c.handle, locs, z, theta, m * m, exa.EXA_FP64, exa.ExaResult())
            assert st == exa.EXA_OK or not ok, seed
            statuses = []
            for ctas in (1, 0):
                out = torch.empty(1, dtype=torch.float64, device="cuda")
                s = torch.empty(1, dtype=torch.int32, device="cuda")
                c.check(exa.exa_ctx_set_batched(c.handle, 64, ctas, 0, 0))
                c.check(exa.exa_loglik_batched(c.handle, 1, [m * m], [locs], [z], to_dev(np.array(theta)), exa.EXA_FP64, out, s))
                statuses.append(int(s.item()))
            assert statuses[1] == exa.EXA_OK or statuses[0] != exa.EXA_OK, seed
