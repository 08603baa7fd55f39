"""The FP64 factorisation on the tensor cores (eight 7-bit digits per value, 512-wide panels) at the edges of its
tiles and panels, against A itself and against the FP64-unit factorisation (a context with 64-wide tiles).

Bound of a factor's residual |L L^T - A|_ij, in units of sqrt(A_ii A_jj) (no row of L exceeds sqrt(A_ii)): each
512-column pass may be off by 512 (2^-55 + 2^-53) 4 = 2,560 u of the two row maxima (u = 2^-53: values rounded at
2^-56 of a row bound that is at most twice the maximum, and the left-out digit products, at most 7 2^-56 + ... <
2^-53), and FP64 rounding in the diagonal blocks and in forming L L^T adds (n + 1) u twice.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def spd(n, seed, exps=0):
    """G G^T + I, symmetrically scaled by powers of two 2^k, |k| <= exps; returns (matrix, scales)."""
    rng = np.random.default_rng(seed)
    g = rng.standard_normal((n, max(2, n // 2))) / np.sqrt(max(2, n // 2))
    a = g @ g.T + np.eye(n)
    a = 0.5 * (a + a.T)
    d = 2.0 ** rng.integers(-exps, exps + 1, n).astype(np.float64)
    return a * d[:, None] * d[None, :], d


def factor(ctx, a, ld):
    import torch
    import paper_1908_06936_gb300 as exa

    n = len(a)
    buf = torch.full((n, ld), 7.0, dtype=torch.float64, device="cuda")  # column j of the matrix is row j here
    buf[:, :n] = torch.as_tensor(a, device="cuda")
    ctx.check(exa.exa_potrf(ctx.handle, buf, n, ld))
    out = buf.cpu().numpy()
    assert np.all(out[:, n:] == 7.0) and np.array_equal(np.tril(out[:, :n], -1), np.tril(a, -1))
    return np.triu(out[:, :n]).T


@pytest.mark.parametrize("n,pad,exps", [(1, 0, 0), (127, 3, 0), (128, 0, 0), (129, 0, 0), (511, 0, 0), (512, 0, 0),
                                        (513, 5, 0), (640, 0, 480), (769, 0, 0), (1024, 0, 0), (1025, 1, 480),
                                        (1664, 0, 0), (2200, 0, 60), (4500, 0, 0)])
def test_factor_residual(n, pad, exps):
    import paper_1908_06936_gb300 as exa

    a, d = spd(n, n, exps)
    root = np.sqrt(np.diag(a) / d / d)
    bound = (-(-n // 512) * 2560 + 2 * (n + 1)) * U * np.outer(root, root)
    with exa.Context(tile_nb=128) as c, exa.Context(tile_nb=64) as general:
        l = factor(c, a, n + pad)
        assert np.array_equal(l, factor(c, a, n + pad))  # repeatable to the bit
        l64 = factor(general, a, n + pad) / d[:, None]
    l = l / d[:, None]
    assert np.all(np.abs(l @ l.T - a / d[:, None] / d[None, :]) <= bound)
    # both factors are exact for matrices within the bound of A, and cond(A) <= 8 here: they agree to a few times it
    assert np.max(np.abs(l - l64)) <= 32 * np.max(bound)


@pytest.mark.parametrize("n,row", [(900, 700), (1300, 511), (1300, 512), (1300, 1299)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -1.0])
def test_failing_pivot_is_reported(n, row, bad):
    import torch
    import paper_1908_06936_gb300 as exa

    a, _ = spd(n, 3)
    if bad < 0:
        a[row, row] = bad
    else:
        a[row, 5] = a[5, row] = bad
    with exa.Context() as c:
        assert exa.exa_potrf(c.handle, torch.as_tensor(a, device="cuda"), n, n) == exa.EXA_ERR_NOT_SPD
        assert exa.exa_last_pivot(c.handle) == row
        good, _ = spd(n, 4)
        c.check(exa.exa_potrf(c.handle, torch.as_tensor(good, device="cuda"), n, n))


def test_workspace_bound_takes_the_fp64_units():
    # 16 MB hold the padded matrix (10.6 MB) and the panels of the FP64-unit factorisation, not the digits
    import paper_1908_06936_gb300 as exa

    a, _ = spd(1100, 5)
    with exa.Context(workspace_bytes=16 << 20) as c, exa.Context() as free:
        l = factor(c, a, 1100)
        assert exa.exa_workspace_bytes(c.handle) <= 16 << 20
        ref = factor(free, a, 1100)
    assert np.max(np.abs(l - ref)) <= 1e-11


@pytest.mark.parametrize("n", [1, 100, 129, 512, 520, 640, 1000, 1025, 1300])
def test_gradient_and_fisher_against_the_fp64_units(n):
    # the bars of the gradient's two forms against each other (1e-10 of the largest component) and of the Fisher
    # information against the oracle (1e-9 of the diagonal)
    import paper_1908_06936_gb300 as exa
    from gpu_util import to_dev
    from paper_1908_06936_gb300 import synth

    theta = (1.2, 0.1, 0.6)
    locs = to_dev(synth.uniform_square(n, n) if n < 4 else synth.jittered_grid(int(np.ceil(np.sqrt(n))), n)[:n])
    z = to_dev(synth.normals(n, n))
    with exa.Context(tile_nb=128) as c, exa.Context(tile_nb=64) as general:
        l, g = c.loglik_grad(locs, z, theta)
        l64, g64 = general.loglik_grad(locs, z, theta)
        f, f64 = c.fisher(locs, theta), general.fisher(locs, theta)
    assert abs(l - l64) <= 1e-10 * abs(l64)
    assert np.all(np.abs(g - g64) <= 1e-10 * max(1.0, float(np.max(np.abs(g64))))), (g, g64)
    assert np.all(np.abs(f - f64) <= 1e-9 * np.sqrt(np.outer(np.diag(f64), np.diag(f64))) + 1e-300), (f, f64)


@pytest.mark.parametrize("n,m", [(1, 1), (100, 65), (512, 64), (513, 63), (640, 2049), (1300, 2500)])
def test_prediction_against_the_fp64_units(n, m):
    # the bars of test_gpu_predict: means to 1e-9 of the largest observation, variances to 1e-9 sigma^2
    import paper_1908_06936_gb300 as exa
    from gpu_util import to_dev
    from paper_1908_06936_gb300 import synth

    theta = (1.2, 0.1, 0.6)
    locs = to_dev(synth.uniform_square(n, n) if n < 4 else synth.jittered_grid(int(np.ceil(np.sqrt(n))), n)[:n])
    z, new = to_dev(synth.normals(n, n)), to_dev(synth.uniform_square(m, m + 1))
    with exa.Context(tile_nb=128) as c, exa.Context(tile_nb=64) as general:
        mean, var = (t.cpu().numpy() for t in c.predict(locs, z, theta, new))
        mean64, var64 = (t.cpu().numpy() for t in general.predict(locs, z, theta, new))
    assert np.all(np.abs(mean - mean64) <= 1e-9 * float(z.abs().max()))
    assert np.all(np.abs(var - var64) <= 1e-9 * theta[0])


def batch(c, ns, tile, ctas, seed=0):
    import torch
    import paper_1908_06936_gb300 as exa
    from gpu_util import to_dev
    from paper_1908_06936_gb300 import synth

    locs = [to_dev(synth.uniform_square(n, seed + r) if n < 4 else
                   synth.jittered_grid(int(np.ceil(np.sqrt(n))), seed + r)[:n]) for r, n in enumerate(ns)]
    z = [to_dev(synth.normals(n, seed + r)) for r, n in enumerate(ns)]
    th = to_dev(synth.theta_perturbations((1.0, 0.1, 0.6), len(ns), seed).ravel())
    out = torch.empty(len(ns), dtype=torch.float64, device="cuda")
    st = torch.empty(len(ns), dtype=torch.int32, device="cuda")
    c.check(exa.exa_ctx_set_batched(c.handle, tile, ctas, 0, 0))
    c.check(exa.exa_loglik_batched(c.handle, len(ns), ns, locs, z, th, exa.EXA_FP64, out, st))
    torch.cuda.synchronize()
    assert np.all(st.cpu().numpy() == 0)
    return out.cpu().numpy()


@pytest.mark.parametrize("ns", [[1], [128, 127], [129, 1, 300, 128, 257], [1000, 400, 401, 129, 2000, 640]])
def test_batched_fp64_against_the_persistent_form(ns):
    # both forms are held to 1e-10 of the oracle elsewhere; a shape change and the persistent form in between leave
    # the tensor-core form's lists right; a context without room for the digits falls back to the persistent form
    import paper_1908_06936_gb300 as exa

    with exa.Context() as c:
        got = batch(c, ns, 0, 0)
        ref = batch(c, ns, 32, 0)
        batch(c, [200] + ns, 0, 0)
        assert np.array_equal(got, batch(c, ns, 0, 0))
    assert np.all(np.abs(got - ref) <= 1e-10 * np.abs(ref))
    with exa.Context() as c:
        batch(c, ns, 64, 1)
        need = exa.exa_workspace_bytes(c.handle)
    with exa.Context(workspace_bytes=need) as c:
        low = batch(c, ns, 0, 0)
        assert exa.exa_workspace_bytes(c.handle) <= need
    assert np.all(np.abs(low - ref) <= 1e-10 * np.abs(ref))


@pytest.mark.parametrize("nrep", [19, 20, 38, 39, 76, 77])
def test_batched_fp64_at_every_cluster_width(nrep):
    # 8, 4, 4, 2, 2 and 1 CTAs a diagonal tile on 152 SMs; the bound of the test above
    import paper_1908_06936_gb300 as exa

    ns = [1 + (37 * r) % 300 for r in range(nrep)]
    with exa.Context() as c:
        got = batch(c, ns, 0, 0)
        ref = batch(c, ns, 32, 0)
    assert np.all(np.abs(got - ref) <= 1e-10 * np.abs(ref))


@pytest.mark.parametrize("m", [23, 40, 64])
def test_mixed_solves_without_room_for_the_block_inverses(m):
    # one byte less than the evaluation holds leaves no room for the 512-wide block inverses: the same factor, solved by
    # the persistent kernels.  Each quadratic form is final to 1e-8 by the refinement's stopping rule.
    import paper_1908_06936_gb300 as exa
    from gpu_util import to_dev
    from paper_1908_06936_gb300 import synth

    locs, z = to_dev(synth.jittered_grid(m, m)), to_dev(synth.normals(m * m, m))
    theta = (1.0, 0.1, 0.5)
    with exa.Context() as c:
        a = c.loglik_ex(locs, z, theta, exa.EXA_MIXED_TF32X3)
        held = exa.exa_workspace_bytes(c.handle)
    with exa.Context(workspace_bytes=held - 1) as c:
        b = c.loglik_ex(locs, z, theta, exa.EXA_MIXED_TF32X3)
        assert exa.exa_workspace_bytes(c.handle) < held
    assert a["logdet"] == b["logdet"]
    assert abs(a["quad"] - b["quad"]) <= 2e-8 * abs(a["quad"])
