"""The FP32 path for D <= 128 (csrc/em_direct.cu): tiles cut to the shape, whole fits enqueued ahead."""
import numpy as np
import pytest
import torch

from oracle import gmm_oracle as orc
from tests.parity_util import assert_stats_close, data_scale

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def fg():
    from paper_2606_10896_b200 import flashgmm

    return flashgmm


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32, device=DEV).contiguous()


def _mixture(N, D, K, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    mu = rng.normal(0, 1.5, (K, D))
    X = mu[rng.integers(0, K, N)] + rng.standard_normal((N, D)) + 3.0
    return (X.astype(np.float32), rng.dirichlet(np.ones(K)).astype(np.float32), (mu + 3.0).astype(np.float32),
            rng.uniform(0.5, 2.0, (K, D)).astype(np.float32))


# component groups of four, blocks of 64, chunks of four dimensions, tiles of 4 to 256 points, lanes that share dimensions
@pytest.mark.parametrize("N,D,K", [(1, 1, 1), (257, 2, 4), (1000, 3, 5), (63, 128, 1), (999, 127, 9), (4097, 31, 16), (300, 33, 17), (20000, 4, 3),
                                   (5000, 100, 63), (4100, 128, 64), (30011, 8, 12), (3000, 6, 65), (2500, 40, 200), (700, 128, 130)])
def test_direct_step_at_the_edges_of_its_tiles(fg, N, D, K):
    X, pi, mu, var = _mixture(N, D, K, N + D + K)
    if K > 2:
        pi[1] = 0.0
    ref = orc.em_step(X, pi, mu, var)
    with fg.Context(0) as c:
        c.gmm_set_path(fg.GMM_PATH_FP32)
        out = [[v.cpu().numpy() if torch.is_tensor(v) else v for v in c.gmm_em_step(_t(X), _t(pi), _t(mu), _t(var))] for _ in range(2)]
        logp, total = c.gmm_score_samples(_t(X), _t(pi), _t(mu), _t(var))
    assert all(np.array_equal(a, b) for a, b in zip(*out))      # the same bits in every run
    assert abs(out[0][3] - ref[3]) <= 1e-5 * abs(ref[3]) + 1e-6 and abs(total - ref[3]) <= 1e-5 * abs(ref[3]) + 1e-6
    assert_stats_close(N, max(1.0, data_scale(X)), out[0][:3], ref[:3], f"N={N} D={D} K={K}")


@pytest.mark.parametrize("isotropic", [False, True])
def test_direct_fit_runs_ahead_and_stops_by_itself(fg, isotropic):
    # more iterations than there are slots for log-likelihoods; then with a tolerance that the fit meets on its way
    X, pi, mu, var = _mixture(3000, 7, 6, 3)
    if isotropic:
        var = np.repeat(var[:, :1], 7, 1)
    step = orc.em_iteration_isotropic if isotropic else orc.em_iteration
    iters, want, p = 150, [], (pi, mu, var)
    for _ in range(iters):
        *p, ll = step(X, *p, 1e-6)[:4]
        want.append(ll)
    want = np.array(want)
    with fg.Context(0) as c:
        c.gmm_set_covariance(fg.GMM_COV_ISOTROPIC if isotropic else fg.GMM_COV_DIAG)
        a = [_t(pi), _t(mu), _t(var)]
        trace, done = c.gmm_fit(_t(X), *a, iters, 1e-6)
        assert done == len(trace) == iters and np.all(np.abs(trace - want) <= 2e-5 * np.abs(want))
        b = [_t(pi), _t(mu), _t(var)]
        short, n = c.gmm_fit(_t(X), *b, iters, 1e-6, tol=1e-6)
        assert 1 < n < iters and np.array_equal(short, trace[:n])
        change = np.abs(np.diff(short)) / np.abs(short[1:])
        assert change[-1] <= 1e-6 and np.all(change[:-1] > 1e-6)
        d = [_t(pi), _t(mu), _t(var)]
        c.gmm_fit(_t(X), *d, n, 1e-6)
        assert all(torch.equal(u, v) for u, v in zip(b, d))      # nothing was done after the iteration that met the tolerance


# A fit that is one launch of a cluster of 16 CTAs: fewer points than CTAs, CTAs without components or with several, lanes per point 1 to 16, dimensions that are no
# multiple of four, rows that do not start on 16 bytes; against steps and updates one by one (the same sums in another order: 1e-4 of the data's scale after
# four iterations at most).
@pytest.mark.parametrize("isotropic", [False, True])
@pytest.mark.parametrize("N,D,K,offset", [(1, 1, 1, 0), (15, 3, 2, 0), (40, 128, 8, 0), (2500, 16, 64, 0), (17, 2, 5, 1), (4099, 31, 9, 1), (1700, 5, 33, 0), (30_000, 2, 2, 0), (900, 1, 17, 3)])
def test_direct_fit_in_one_launch(fg, N, D, K, offset, isotropic):
    X, pi, mu, var = _mixture(N, D, K, 7 * N + D + K)
    var = np.maximum(var, 1.0)
    if isotropic:
        var = np.repeat(var[:, :1], D, 1)
    if K > 2:
        pi[1] = 0.0                                        # (an empty component keeps its mean and variance)
    flat = torch.empty(N * D + offset, device=DEV)
    Xd = flat[offset:].view(N, D)
    Xd.copy_(_t(X))
    with fg.Context(0) as c:
        c.gmm_set_path(fg.GMM_PATH_FP32)
        c.gmm_set_covariance(fg.GMM_COV_ISOTROPIC if isotropic else fg.GMM_COV_DIAG)
        a, b, want = [_t(pi), _t(mu), _t(var)], [_t(pi), _t(mu), _t(var)], []
        for _ in range(4):
            Nk, S1, S2, ll = c.gmm_em_step(Xd, *a)
            want.append(ll)
            (c.gmm_finalize_isotropic if isotropic else c.gmm_finalize)(N, Nk, S1, S2, 0.3, *a)
        counts = c.gmm_update_counts()
        before = c.gmm_launch_count()
        trace, done = c.gmm_fit(Xd, *b, 4, 0.3)
        assert c.gmm_launch_count() - before <= 2 and done == 4 and c.gmm_update_counts() == counts
        assert np.all(np.abs(trace - want) <= 1e-5 * np.abs(want) + 1e-5)
        for u, v, s in zip(b, a, (1.0, data_scale(X) if N > 1 else 1.0, 1.0)):
            assert float((u - v).abs().max()) <= 1e-4 * max(s, 1.0)
        again = [_t(pi), _t(mu), _t(var)]
        c.gmm_fit(Xd, *again, 4, 0.3)
        assert all(torch.equal(u, v) for u, v in zip(again, b))      # the same bits in every run


# Sums of many terms are taken in parts.  Points far from two components that share them: a quadratic form q errs by 2^-24 q times a factor that grows with the root of the
# terms added one after the other (1.15 and 1.26 in parts at the two widths, 1.48 and 1.83 in one sum; the line is between them), a responsibility by that times r (1 - r).
@pytest.mark.parametrize("D", [60, 100])
def test_direct_fit_in_one_launch_far_from_two_components(fg, D):
    rng = np.random.default_rng(D)
    N = 2500
    mu = np.stack([np.full(D, -0.01), np.full(D, 0.01)]).astype(np.float32)
    var = rng.uniform(0.5, 2.0, (1, D)).repeat(2, 0).astype(np.float32)
    pi = np.full(2, 0.5, np.float32)
    X = (30.0 * rng.standard_normal((N, D))).astype(np.float32)
    x = X.astype(np.float64)
    q = 0.5 * ((x[:, None] - mu) ** 2 / var).sum(2)
    r = 1.0 / (1.0 + np.exp(q - q[:, ::-1]))
    n = r.sum(0)
    m = r.T @ x / n[:, None]
    with fg.Context(0) as c:
        c.gmm_set_path(fg.GMM_PATH_FP32)
        p = [_t(pi), _t(mu), _t(var)]
        before = c.gmm_launch_count()
        c.gmm_fit(_t(X), *p, 1, 1e-6)
        assert c.gmm_launch_count() - before == 1
    err = np.sqrt(((p[1].cpu().numpy() - m) ** 2).mean())
    unit = 2.0 ** -24 * np.sqrt((((q * r * r[:, ::-1])[:, :, None] * x[:, None]) ** 2).sum(0) / n[:, None] ** 2).mean()
    assert err <= np.sqrt(D / 42) * unit


# Points of one component each, B standard deviations from the centre that the sums are taken about: (x - g)^2 is B^2 times the variance.  A thread adds up L rows, 4 at a time: 2^-24 of
# the sums so far for each addition are in all 2^-24 sqrt(N / 2 (4^2 / 3 + L^2 / (3 x 4))) of one row (one sum of all: L^2 / 3), random signs, here with a fifth to spare.
@pytest.mark.parametrize("N,D", [(3000, 128), (7500, 64)])
def test_direct_fit_in_one_launch_far_from_its_centre(fg, N, D):
    rng = np.random.default_rng(N)
    B = 30.0
    mu = np.stack([np.full(D, -B), np.full(D, B)]).astype(np.float32)
    var, pi = np.ones((2, D), np.float32), np.full(2, 0.5, np.float32)
    c = np.arange(N) % 2
    X = (mu[c] + rng.standard_normal((N, D))).astype(np.float32)
    v = np.stack([X[c == k].astype(np.float64).var(0) for k in (0, 1)])
    with fg.Context(0) as ctx:
        ctx.gmm_set_path(fg.GMM_PATH_FP32)
        p = [_t(pi), _t(mu), _t(var)]
        before = ctx.gmm_launch_count()
        ctx.gmm_fit(_t(X), *p, 1, 1e-6)
        assert ctx.gmm_launch_count() - before == 1
    err = np.sqrt((((p[2].cpu().numpy() - v) / v) ** 2).mean())
    L = -(-(-(-N // 16)) // (512 // (D // 4)))             # (rows of a CTA, threads for the same four dimensions)
    assert err <= 1.2 * 2.0 ** -24 * B * B / np.sqrt(N / 2) * np.sqrt(16 / 3 + L * L / 12)


# Fits of mixtures with K D <= 1024 are one launch for as many iterations as there are slots for log-likelihoods (63 ahead), others the launches of every iteration
@pytest.mark.parametrize("isotropic", [False, True])
@pytest.mark.parametrize("N,D,K", [(3000, 7, 6), (3000, 24, 48)])
def test_direct_fit_over_more_iterations_than_slots(fg, N, D, K, isotropic):
    X, pi, mu, var = _mixture(N, D, K, 3)
    if isotropic:
        var = np.repeat(var[:, :1], D, 1)
    step = orc.em_iteration_isotropic if isotropic else orc.em_iteration
    iters, want, p = 150, [], (pi, mu, var)
    for _ in range(iters):
        *p, ll = step(X, *p, 1e-6)[:4]
        want.append(ll)
    want = np.array(want)
    with fg.Context(0) as c:
        c.gmm_set_path(fg.GMM_PATH_FP32)
        c.gmm_set_covariance(fg.GMM_COV_ISOTROPIC if isotropic else fg.GMM_COV_DIAG)
        a = [_t(pi), _t(mu), _t(var)]
        before = c.gmm_launch_count()
        trace, done = c.gmm_fit(_t(X), *a, iters, 1e-6)
        launches = c.gmm_launch_count() - before
        assert launches > 2 * iters if K * D > 1024 else launches == 3
        assert done == len(trace) == iters and np.all(np.abs(trace - want) <= 2e-5 * np.abs(want))
        b = [_t(pi), _t(mu), _t(var)]
        short, n = c.gmm_fit(_t(X), *b, iters, 1e-6, tol=1e-6)
        assert 1 < n < iters and np.array_equal(short, trace[:n])
        change = np.abs(np.diff(short)) / np.abs(short[1:])
        assert change[-1] <= 1e-6 and np.all(change[:-1] > 1e-6)
        d = [_t(pi), _t(mu), _t(var)]
        c.gmm_fit(_t(X), *d, n, 1e-6)
        assert all(torch.equal(u, v) for u, v in zip(b, d))      # nothing was done after the iteration that met the tolerance


# The launches of every iteration against steps and updates one by one: parameters, counts of the updates, the same bits in every run.
@pytest.mark.parametrize("isotropic", [False, True])
@pytest.mark.parametrize("N,D,K,offset", [(40, 128, 9, 0), (1700, 33, 37, 1), (2500, 17, 64, 0)])
def test_direct_fit_beyond_one_launch(fg, N, D, K, offset, isotropic):
    X, pi, mu, var = _mixture(N, D, K, 7 * N + D + K)
    var = np.maximum(var, 1.0)
    if isotropic:
        var = np.repeat(var[:, :1], D, 1)
    pi[1] = 0.0                                            # (an empty component keeps its mean and variance)
    flat = torch.empty(N * D + offset, device=DEV)
    Xd = flat[offset:].view(N, D)
    Xd.copy_(_t(X))
    with fg.Context(0) as c:
        c.gmm_set_path(fg.GMM_PATH_FP32)
        c.gmm_set_covariance(fg.GMM_COV_ISOTROPIC if isotropic else fg.GMM_COV_DIAG)
        a, b, want = [_t(pi), _t(mu), _t(var)], [_t(pi), _t(mu), _t(var)], []
        for _ in range(4):
            Nk, S1, S2, ll = c.gmm_em_step(Xd, *a)
            want.append(ll)
            (c.gmm_finalize_isotropic if isotropic else c.gmm_finalize)(N, Nk, S1, S2, 0.3, *a)
        counts = c.gmm_update_counts()
        before = c.gmm_launch_count()
        trace, done = c.gmm_fit(Xd, *b, 4, 0.3)
        assert c.gmm_launch_count() - before > 8 and done == 4 and c.gmm_update_counts() == counts
        assert np.all(np.abs(trace - want) <= 1e-5 * np.abs(want) + 1e-5)
        for u, v, s in zip(b, a, (1.0, data_scale(X), 1.0)):
            assert float((u - v).abs().max()) <= 1e-4 * max(s, 1.0)
        again = [_t(pi), _t(mu), _t(var)]
        c.gmm_fit(Xd, *again, 4, 0.3)
        assert all(torch.equal(u, v) for u, v in zip(again, b))


def test_direct_fit_beyond_one_launch_keeps_the_parameters_of_a_step_that_fails(fg):
    X, pi, mu, var = _mixture(900, 24, 48, 9)
    X[17, 2] = np.nan
    with fg.Context(0) as c:
        c.gmm_set_path(fg.GMM_PATH_FP32)
        a = [_t(pi), _t(mu), _t(var)]
        with pytest.raises(fg.GmmError):
            c.gmm_fit(_t(X), *a, 5, 1e-6)
        assert all(np.array_equal(u.cpu().numpy(), v) for u, v in zip(a, (pi, mu, var)))


def test_direct_fit_keeps_the_parameters_of_a_step_that_fails(fg):
    X, pi, mu, var = _mixture(500, 5, 4, 9)
    X[17, 2] = np.nan
    with fg.Context(0) as c:
        a = [_t(pi), _t(mu), _t(var)]
        with pytest.raises(fg.GmmError):
            c.gmm_fit(_t(X), *a, 5, 1e-6)
        assert all(np.array_equal(u.cpu().numpy(), v) for u, v in zip(a, (pi, mu, var)))


@pytest.mark.parametrize("N,D,K", [(999, 112, 65), (999, 113, 65), (1000, 128, 64), (1, 113, 65), (4097, 127, 200), (65_537 + 64, 128, 66)])
def test_fp32_step_on_either_side_of_the_fixed_tiles(fg, N, D, K):
    X, pi, mu, var = _mixture(N, D, K, N + D + K)
    ref = orc.em_step(X, pi, mu, var)
    with fg.Context(0) as c:
        c.gmm_set_path(fg.GMM_PATH_FP32)
        got = [v.cpu().numpy() if torch.is_tensor(v) else v for v in c.gmm_em_step(_t(X), _t(pi), _t(mu), _t(var))]
        logp, total = c.gmm_score_samples(_t(X), _t(pi), _t(mu), _t(var))
    assert abs(got[3] - ref[3]) <= 1e-5 * abs(ref[3]) + 1e-6 and abs(total - ref[3]) <= 1e-5 * abs(ref[3]) + 1e-6
    assert_stats_close(N, max(1.0, data_scale(X)), got[:3], ref[:3], f"N={N} D={D} K={K}")
