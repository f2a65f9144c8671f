"""The screening path for D <= 128 (csrc/em_screen.cu): one tensor sweep over a single fp16 product marks the (point,
component) pairs that can matter, those are evaluated exactly.  GMM_PATH_AUTO tries it first; gmm_last_exact_count is the
number of components with a weight after a step that took it."""
import numpy as np
import pytest
import torch

from oracle import gmm_oracle as orc
from paper_2606_10896_b200 import synth
from tests.parity_util import assert_stats_close, data_scale

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def fg():
    from paper_2606_10896_b200 import flashgmm

    return flashgmm


def _t(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device=DEV).contiguous()


def _mixture(N, D, K, seed, collapsed=0):
    """Separate clusters; some components share a cluster, the last ``collapsed`` ones sit on single points."""
    rng = np.random.Generator(np.random.PCG64(seed))
    centre = rng.normal(0, 3, (K, D))
    centre[1::7] = centre[0::7][: len(centre[1::7])] + 0.3 * rng.normal(size=(len(centre[1::7]), D))
    std = rng.uniform(0.5, 1.5, (K, D))
    c = rng.integers(0, K, N)
    X = (centre[c] + std[c] * rng.standard_normal((N, D))).astype(np.float32)
    mu, var = centre + 0.2 * rng.normal(size=(K, D)), std ** 2
    if collapsed:
        mu[-collapsed:] = X[rng.integers(0, N, collapsed)]
        var[-collapsed:] = 1e-6
    pi = rng.dirichlet(np.ones(K))
    return X, pi.astype(np.float32), mu.astype(np.float32), var.astype(np.float32)


def _step(fg, c, X, pi, mu, var, expect_count, what):
    ref = orc.em_step(X, pi, mu, var)
    out = []
    for _ in range(2):
        Nk, S1, S2, L = c.gmm_em_step(_t(X), _t(pi), _t(mu), _t(var))
        out.append((Nk.cpu().numpy(), S1.cpu().numpy(), S2.cpu().numpy(), L))
    if expect_count is not None:
        assert c.gmm_last_path() == fg.GMM_PATH_TENSOR and c.gmm_last_exact_count() == expect_count, what
    assert abs(out[0][3] - ref[3]) <= 1e-5 * abs(ref[3]) + 1e-6, what
    assert_stats_close(len(X), max(1.0, data_scale(X)), out[0][:3], ref[:3], what)
    for a, b in zip(out[0], out[1]):                       # the same bits in every run
        assert np.array_equal(a, b), what


# tiles of 256 points, ranges of 512, atoms of 32 dimensions, k-steps of 8, groups of 128 and blocks of 32 components
@pytest.mark.parametrize("N,D,K", [(1, 8, 64), (255, 128, 64), (257, 33, 65), (511, 31, 128), (513, 32, 129), (1024, 97, 257),
                                   (1500, 41, 1000), (1300, 9, 90), (1500, 24, 16), (2049, 128, 48), (3001, 127, 96), (700, 64, 4096), (2049, 100, 160)])
def test_screen_against_oracle_at_the_edges_of_its_tiles(fg, monkeypatch, N, D, K):
    monkeypatch.setenv("GMM_SCREEN_MARKS", "1000")
    X, pi, mu, var = _mixture(N, D, K, N + D + K, collapsed=3)
    pi[K // 2] = 0.0                                       # one component without a weight
    with fg.Context(0) as c:
        _step(fg, c, X, pi, mu, var, K - 1, f"screen N={N} D={D} K={K}")


# The sweep converts X itself (D > 64; D > 32 up to K = 512; any D up to K = 256) in chunks of 32 to 256 rows, by bulk copies that start
# at 16-byte boundaries: X at any offset of 4 bytes, rows that are no multiple of 16 bytes, ragged last chunks, either side of the rule.
@pytest.mark.parametrize("offset", [0, 1, 3])
@pytest.mark.parametrize("N,D,K", [(31, 128, 64), (255, 99, 64), (289, 100, 130), (1055, 97, 64), (545, 65, 96), (577, 48, 512), (577, 48, 513), (320, 36, 64), (513, 72, 2049), (513, 32, 256), (513, 31, 257), (800, 9, 64)])
def test_screen_takes_its_rows_from_anywhere(fg, monkeypatch, N, D, K, offset):
    monkeypatch.setenv("GMM_SCREEN_MARKS", "1000")
    X, pi, mu, var = _mixture(N, D, K, 3 * N + D + K, collapsed=1)
    off = (11.0 * (np.arange(D) % 5 - 1)).astype(np.float32)   # (a mean of its own in every dimension)
    X, mu = X + off, mu + off
    X[N // 2, D - 1] = 4000.0                              # beyond the range of the 16-bit rows: evaluated in full
    ref = orc.em_step(X, pi, mu, var)
    flat = torch.empty(N * D + offset, dtype=torch.float32, device=DEV)
    Xd = flat[offset:].view(N, D)
    Xd.copy_(_t(X))
    with fg.Context(0) as c:
        Nk, S1, S2, L = c.gmm_em_step(Xd, _t(pi), _t(mu), _t(var))
        assert c.gmm_last_path() == fg.GMM_PATH_TENSOR and c.gmm_last_exact_count() == K
    assert abs(L - ref[3]) <= 1e-5 * abs(ref[3])
    assert_stats_close(N, max(1.0, data_scale(X)), (Nk.cpu().numpy(), S1.cpu().numpy(), S2.cpu().numpy()), ref[:3], f"N={N} D={D} K={K} offset={offset}")


# The bounds are in the data's own units about the mixture's mean, so moving data and mixture by the same vector changes no verdict.  Numbers of
# chunks of eight dimensions that are no power of two (2, 3, 5, 9, 13), where a row has lanes without dimensions.
@pytest.mark.parametrize("D", [9, 20, 40, 72, 100])
def test_screen_takes_data_that_are_not_about_zero(fg, D):
    N, K = 3000, 64
    rng = np.random.default_rng(D)
    centre = rng.normal(0, max(3.0, 30 / D ** 0.5), (K, D))
    X0 = centre[rng.integers(0, K, N)] + rng.normal(size=(N, D))
    pi, var = np.full(K, 1 / K, np.float32), np.ones((K, D), np.float32)
    with fg.Context(0) as c:
        def launches(call):
            before = c.gmm_launch_count()
            out = call()
            return c.gmm_launch_count() - before, out

        counts = []
        for shift in (0.0, 30.0, -30.0, 1000.0):
            X, mu = (X0 + shift).astype(np.float32), (centre + shift).astype(np.float32)
            ref = orc.em_step(X, pi, mu, var)
            n, got = launches(lambda: c.gmm_em_step(_t(X), _t(pi), _t(mu), _t(var)))
            assert c.gmm_last_exact_count() == K, shift
            counts.append((n, launches(lambda: c.gmm_kmeans_step(_t(X), _t(mu)))[0], launches(lambda: c.gmm_score_samples(_t(X), _t(pi), _t(mu), _t(var)))[0]))
            assert abs(got[3] - ref[3]) <= 1e-5 * abs(ref[3])
            assert_stats_close(N, data_scale(X), [v.cpu().numpy() for v in got[:3]], ref[:3], f"D={D} shift={shift}")
        assert len(set(counts)) == 1, counts
        X[7, 0] = np.inf                                   # (what a k-means step that goes on to the dense kernels launches)
        before = c.gmm_launch_count()
        with pytest.raises(fg.GmmError):
            c.gmm_kmeans_step(_t(X), _t(mu))
        assert c.gmm_launch_count() - before > counts[0][1]


def test_screen_accumulates_over_pieces_and_takes_unaligned_rows(fg, monkeypatch):
    monkeypatch.setenv("GMM_SCREEN_MARKS", "1000")
    monkeypatch.setenv("GMM_SCREEN_PIECE", "768")
    X, pi, mu, var = _mixture(3000, 66, 130, 5, collapsed=2)
    with fg.Context(0) as c:
        _step(fg, c, X, pi, mu, var, 130, "four pieces, rows of 8-byte alignment")
        host = c.gmm_em_step_host(X, pi, mu, var)
        dev = c.gmm_em_step(_t(X), _t(pi), _t(mu), _t(var))
        assert np.array_equal(host[0], dev[0].cpu().numpy()) and np.array_equal(host[2], dev[2].cpu().numpy()) and host[3] == dev[3]


def test_screen_rows_without_a_list(fg, monkeypatch):
    """A few points far outside the range of the fp16 plane, and a few that a great many components explain about equally well:
    both leave the sweep without a list and are evaluated against all components."""
    monkeypatch.setenv("GMM_SCREEN_MARKS", "1000")
    N, D, K = 6000, 24, 700
    X, pi, mu, var = _mixture(N, D, K, 11)
    X[::1500] = 4000.0                                     # beyond 240 times the data's spread
    mu[100:], var[100:] = 6.0 + 0.05 * mu[100:], 1.0       # 600 components in one place ...
    rows = np.setdiff1d(np.arange(N), np.arange(0, N, 1500))
    X[rows] = (mu[rows % 100] + np.sqrt(var[rows % 100])).astype(np.float32)
    X[100::1000] = 6.0                                     # ... and six points there
    with fg.Context(0) as c:
        _step(fg, c, X, pi, mu, var, K, "rows without a list")


def test_screen_leaves_broad_posteriors_to_the_dense_kernels(fg):
    rng = np.random.default_rng(3)
    N, D, K = 4000, 16, 128
    X = rng.normal(size=(N, D)).astype(np.float32)
    mu = (0.1 * rng.normal(size=(K, D))).astype(np.float32)
    var = rng.uniform(0.8, 1.2, (K, D)).astype(np.float32)
    pi = np.full(K, 1 / K, np.float32)
    with fg.Context(0) as c:
        _step(fg, c, X, pi, mu, var, None, "broad posteriors")
        assert c.gmm_last_path() == fg.GMM_PATH_TENSOR and c.gmm_last_exact_count() < K
        # a fit applies every iteration's update exactly once, whichever kernels took the step
        p, m, v = _t(pi), _t(mu), _t(var)
        trace, done = c.gmm_fit(_t(X), p, m, v, 3)
        ref = orc.fit(X, pi, mu, var, 3, var_floor=1e-6)
        assert done == 3
        np.testing.assert_allclose(trace, ref["trace"], rtol=1e-5)


def test_screen_reports_non_finite_data(fg):
    X, pi, mu, var = _mixture(2000, 40, 128, 3)
    X[1234, 5] = np.nan
    with fg.Context(0) as c:
        with pytest.raises(fg.GmmError) as e:
            c.gmm_em_step(_t(X), _t(pi), _t(mu), _t(var))
        assert e.value.code == fg.GMM_ENUMERIC
        X[1234, 5] = 0.0
        c.gmm_em_step(_t(X), _t(pi), _t(mu), _t(var))


def test_screen_wait_that_runs_out(fg, monkeypatch):
    """One CTA of the sweep keeps back the arrival that its other warps wait for.  Their waits run out (2 s), the kernel ends by itself,
    nothing reads the lists that it has not written, and the call - the next synchronising one after an assignment - says so."""
    X, pi, mu, var = _mixture(3000, 40, 200, 8)
    ref = orc.em_step(X, pi, mu, var)
    monkeypatch.setenv("GMM_SCREEN_MARKS", "1000")
    monkeypatch.setenv("GMM_SCREEN_TEST_SILENT", "2")
    with fg.Context(0) as c:
        for call in (lambda: c.gmm_em_step(_t(X), _t(pi), _t(mu), _t(var)), lambda: c.gmm_kmeans_step(_t(X), _t(mu)),
                     lambda: (c.gmm_assign_topm(_t(X), _t(pi), _t(mu), _t(var), 2), c.gmm_sync_status())):
            with pytest.raises(fg.GmmError) as e:
                call()
            assert e.value.code == fg.GMM_ETIMEOUT
        c.gmm_sync_status()
    monkeypatch.delenv("GMM_SCREEN_TEST_SILENT")
    with fg.Context(0) as c:
        got = c.gmm_em_step(_t(X), _t(pi), _t(mu), _t(var))
        assert abs(got[3] - ref[3]) <= 1e-5 * abs(ref[3])


def test_screen_leaves_non_finite_data_to_the_fp32_kernels(fg, monkeypatch):
    """K < 64: the assignment and the k-means step take such data as the FP32 kernels do, with or without the screening sweep in front."""
    X, pi, mu, var = _mixture(3000, 40, 48, 4)
    bad, cen = X.copy(), mu.copy()
    bad[1234, 5], bad[2000] = np.nan, np.inf
    cen[7, 3] = np.nan
    got = []
    for marks in ("1000", "0"):
        monkeypatch.setenv("GMM_SCREEN_MARKS", marks)
        with fg.Context(0) as c:
            idx, resp = c.gmm_assign_topm(_t(bad), _t(pi), _t(mu), _t(var), 1)
            c.gmm_sync_status()
            a, new, counts, inertia = c.gmm_kmeans_step(_t(bad), _t(mu))
            b, newer, _, _ = c.gmm_kmeans_step(_t(X), _t(cen))
            got.append([v.cpu().numpy() for v in (idx, resp, a, new, counts, b, newer)] + [inertia])
    for u, v in zip(*got):
        assert np.array_equal(u, v, equal_nan=True)


def test_config2_free_running_through_the_screening_path(fg):
    spec = synth.CONFIGS[2].with_n(20_000)
    X = synth.sample_host(spec)
    pi0, mu0, var0 = synth.init_params(X, spec)
    ref = orc.fit(X, pi0, mu0, var0, 8, var_floor=spec.var_floor)
    with fg.Context(0) as c:
        trace, done = c.gmm_fit(_t(X), _t(pi0), _t(mu0), _t(var0), 8, spec.var_floor)
        assert done == 8
        np.testing.assert_allclose(trace, ref["trace"], rtol=1e-4)


# the other entry points on the path, in pieces of 768 points: several tiles and pieces, a last piece of one point, groups that are
# empty, larger than a piece, or share one
@pytest.mark.parametrize("N,D,K", [(1, 16, 64), (3073, 40, 100), (2500, 128, 1024), (4000, 9, 300), (900, 66, 4096), (3000, 33, 31)])
def test_screen_kmeans_scores_and_fisher_vectors(fg, monkeypatch, N, D, K):
    from oracle.fisher import fisher_vectors
    from oracle.kmeans import kmeans_step

    monkeypatch.setenv("GMM_SCREEN_MARKS", "1000")
    monkeypatch.setenv("GMM_SCREEN_PIECE", "768")
    X, pi, mu, var = _mixture(N, D, K, N + D + K)
    offsets = np.array([0, N // 8, N // 8, N // 8 + N // 16, N - N // 5, N], np.int64)
    lz = orc.responsibilities(X, pi, mu, var)[1]
    G_ref = fisher_vectors(X, offsets, pi, mu, var)
    a_r, new_r, _, inertia_r, gap = kmeans_step(X, mu.astype(np.float64))
    runs = []
    with fg.Context(0) as c:
        for _ in range(2):
            logp, total = c.gmm_score_samples(_t(X), _t(pi), _t(mu), _t(var))
            G, ll = c.gmm_fisher_vectors(_t(X), offsets, _t(pi), _t(mu), _t(var))
            a, new, counts, inertia = c.gmm_kmeans_step(_t(X), _t(mu))
            runs.append((logp.cpu().numpy(), total, G.cpu().numpy(), ll, a.cpu().numpy(), new.cpu().numpy(), counts.cpu().numpy(), inertia))
    for u, v in zip(*runs):
        assert np.array_equal(u, v)                            # the same bits in every run
    logp, total, G, ll, a, new, counts, inertia = runs[0]
    assert np.all(np.abs(logp - lz) <= 1e-5 * np.abs(lz) + 1e-4) and abs(total - lz.sum()) <= 1e-5 * abs(lz.sum())
    assert abs(ll - lz.sum()) <= 1e-5 * abs(lz.sum())
    assert np.abs(G - G_ref).max() <= 2e-5 * (1 + np.abs(G_ref).max()) and np.all(G[1] == 0.0)
    tie = gap <= 1e-4 * D * float(X.astype(np.float64).var(0).mean() if N > 1 else 1.0)
    assert np.all((a == a_r) | tie) and counts.sum() == N and np.array_equal(counts, np.bincount(a, minlength=K))
    assert abs(inertia - inertia_r) <= 1e-5 * abs(inertia_r)
    for k in np.unique(a)[:50]:
        np.testing.assert_allclose(new[k], X[a == k].astype(np.float64).mean(0), rtol=0, atol=1e-5)
    empty = np.setdiff1d(np.arange(K), a)
    assert np.array_equal(new[empty], mu[empty])               # a centroid without points stays where it is


# Sums per group and component: a warp has a run of one to eight components (of few groups with many points one, of many small groups eight; the last run of a
# group fewer), empty groups and components, pairs of one component beyond a stage of 4 to 32 rows; X at 4 bytes past a boundary.
@pytest.mark.parametrize("G,most,D,K,offset", [(600, 60, 33, 50, 0), (600, 50, 20, 50, 0), (500, 40, 128, 64, 0), (450, 60, 64, 70, 1), (5, 2500, 9, 20, 0), (3, 3000, 100, 33, 0), (700, 30, 8, 48, 0)])
def test_screen_sums_per_group(fg, monkeypatch, G, most, D, K, offset):
    from oracle.fisher import fisher_vectors

    monkeypatch.setenv("GMM_SCREEN_MARKS", "1000")
    rng = np.random.default_rng(G + D + K)
    size = rng.integers(0, most, G)
    size[0] += 1
    offsets = np.concatenate([[0], np.cumsum(size)]).astype(np.int64)
    N = int(offsets[-1])
    X, pi, mu, var = _mixture(N, D, K, G + D)
    pi[K // 2] = 0.0
    flat = torch.empty(N * D + offset, device=DEV)
    Xd = flat[offset:].view(N, D)
    Xd.copy_(_t(X))
    lz = orc.responsibilities(X, pi, mu, var)[1]
    ref = fisher_vectors(X, offsets, pi, mu, var)
    with fg.Context(0) as c:
        F, ll = c.gmm_fisher_vectors(Xd, offsets, _t(pi), _t(mu), _t(var))
        again = c.gmm_fisher_vectors(Xd, offsets, _t(pi), _t(mu), _t(var))
        assert c.gmm_last_exact_count() == K - 1
    assert torch.equal(F, again[0]) and ll == again[1] and abs(ll - lz.sum()) <= 1e-5 * abs(lz.sum())
    F = F.cpu().numpy()
    assert np.abs(F - ref).max() <= 2e-5 * (1 + np.abs(ref).max()) and np.all(F[size == 0] == 0.0)


# One group of 32768 points on two components: sums over n of 12000 pairs and more.  32 of them at a time are added to a running fp32 sum, n / 32 additions that each err by
# at most 2^-24 of what the sum has reached: as random signs, 2^-24 sqrt(n / 32) / 3 of the whole (a third: the sum grows linearly, errors are spread evenly).  On separate clusters
# sum r (x - mu)^2 / (n var) is 1 + sqrt(2 pi) T G_sigma / n.  (Eight pairs at a time would be twice that, four 2.8 times.)
@pytest.mark.parametrize("D", [128, 64, 100])
def test_screen_sums_of_a_large_group(fg, monkeypatch, D):
    from oracle.fisher import fisher_vectors

    monkeypatch.setenv("GMM_SCREEN_MARKS", "1000")
    rng = np.random.default_rng(D)
    T, K = 32768, 20
    pi = np.full(K, 0.001, np.float32)
    pi[:2] = 0.982 * np.array([0.6, 0.4])
    mu = rng.normal(0, 3, (K, D)).astype(np.float32)
    var = rng.uniform(0.5, 1.5, (K, D)).astype(np.float32)
    c = (np.arange(T) % 5 < 2).astype(int)
    X = (mu[c] + np.sqrt(var)[c] * rng.standard_normal((T, D))).astype(np.float32)
    offsets = np.array([0, T], np.int64)
    ref = fisher_vectors(X, offsets, pi, mu, var)
    with fg.Context(0) as ctx:
        F = ctx.gmm_fisher_vectors(_t(X), offsets, _t(pi), _t(mu), _t(var))[0].cpu().numpy()
        assert ctx.gmm_last_exact_count() == K
    n = np.bincount(c)
    err = np.sqrt(((F - ref)[0, 1, :2] ** 2).mean(1)) * np.sqrt(2.0 * pi[:2]) * T / n
    assert np.all(err <= 2.0 ** -24 * np.sqrt(n / 32) / 3)


# Every point has a second component with a share of 1e-8 or so of it, which 32-bit sums of a component's weights lose: so the log-likelihood is that of the points, one by one, and
# no product of the components' sums.  Roundings of the points' own values go either way and are gone in the sum (what all points of a component lose alike is added back).  Those
# of the K D / 2 different weights 1 / (2 var) stay: 2^-25 / sqrt(3) each, of half a unit per dimension in 1.5 per dimension; four standard deviations of them.
@pytest.mark.parametrize("N,D,K", [(60_000, 64, 128), (32_768, 128, 64), (250_000, 16, 96)])
def test_screen_log_likelihood_of_shared_points(fg, monkeypatch, N, D, K):
    monkeypatch.setenv("GMM_SCREEN_MARKS", "1000")
    rng = np.random.default_rng(N + D)
    mu = rng.normal(0, 6, (K, D))
    step = rng.standard_normal((K // 2, D))
    mu[1::2] = mu[::2] + 6.0 * step / np.linalg.norm(step, axis=1, keepdims=True)
    var = np.repeat(rng.uniform(0.8, 1.2, (K // 2, D)), 2, 0)
    c = rng.integers(0, K, N)
    X = _t(mu[c] + np.sqrt(var)[c] * rng.standard_normal((N, D)))
    pi, mu, var = _t(np.full(K, 1.0 / K)), _t(mu), _t(var)
    x, m, v = X.double(), mu.double(), var.double()
    own = torch.as_tensor(c, device=DEV)
    two = torch.stack([-0.5 * ((x - m[own ^ i]) ** 2 / v[own] + (2 * np.pi * v[own]).log()).sum(1) for i in (0, 1)], 1)      # (all others: below 2^-40)
    want = float((torch.logsumexp(two, 1) + pi.double()[0].log()).sum())
    with fg.Context(0) as ctx:
        err = [abs(ctx.gmm_em_step(X, pi, mu, var)[3] - want) / abs(want)]
        assert ctx.gmm_last_exact_count() == K
        offsets = np.append(np.arange(0, N, 20_000), N).astype(np.int64)
        err.append(abs(ctx.gmm_fisher_vectors(X, offsets, pi, mu, var)[1] - want) / abs(want))
        assert ctx.gmm_last_exact_count() == K
    assert max(err) <= 4 * 2.0 ** -25 / np.sqrt(3) / 3 * np.sqrt(2 / (K * D))


# Beyond 200,000 points the evaluation sorts a CTA's points by their marks.  A point's values do not depend on the points it is worked on with, so they are
# the same bits as from two calls that do not sort.  Every other point has 24 marks: 32 of those together have more than a warp has room for at a time.
@pytest.mark.parametrize("N,D,K,offset", [(200_001, 128, 96, 0), (200_100, 100, 64, 0), (213_121, 64, 1100, 0), (231_000, 24, 2100, 0), (200_193, 32, 64, 1), (200_031, 9, 64, 0)])
def test_screen_values_are_those_of_smaller_calls(fg, monkeypatch, N, D, K, offset):
    monkeypatch.setenv("GMM_SCREEN_MARKS", "1000")
    gen = torch.Generator(device=DEV).manual_seed(N + D)
    mu = 12.0 / D ** 0.5 * torch.randn((K, D), device=DEV, generator=gen) * (1 + 8 / D)
    mu[1:24] = mu[0] + 0.05 * torch.randn((23, D), device=DEV, generator=gen)
    c = torch.randint(24, K, (N,), device=DEV, generator=gen)
    c[::2] = torch.randint(0, 24, (len(c[::2]),), device=DEV, generator=gen)
    flat = torch.empty(N * D + offset, device=DEV)
    X = flat[offset:].view(N, D)
    X.copy_(mu[c] + torch.randn((N, D), device=DEV, generator=gen))
    pi, var = torch.full((K,), 1.0 / K, device=DEV), torch.ones((K, D), device=DEV)
    cut = 390 * 256                                        # (whole tiles: which rows find no room in a tile's lists is not for the comparison)
    with fg.Context(0) as ctx:
        def call(x):
            before = ctx.gmm_launch_count()
            logp, _ = ctx.gmm_score_samples(x, pi, mu, var)
            assert ctx.gmm_launch_count() - before < 12                # (nothing was left to the dense kernels)
            idx, resp = ctx.gmm_assign_topm(x, pi, mu, var, 2)
            near = ctx.gmm_kmeans_step(x, mu)[0]
            return logp, idx, resp, near

        whole, head, rest = call(X), call(X[:cut]), call(X[cut:])
        for w, a, b in zip(whole, head, rest):
            assert torch.equal(w, torch.cat([a, b]))
        Nk, S1, S2, L = ctx.gmm_em_step(X, pi, mu, var)
        assert ctx.gmm_last_exact_count() == K
        assert abs(float(Nk.sum()) - N) <= 1e-6 * N and abs(L - float(whole[0].double().sum())) <= 1e-6 * abs(L)
        again = ctx.gmm_em_step(X, pi, mu, var)
        assert again[3] == L and all(torch.equal(a, b) for a, b in zip(again[:3], (Nk, S1, S2)))


# the top-m assignment through the sweep: a point far away from everything, components without a weight (fewer than m with one, once)
@pytest.mark.parametrize("N,D,K,m", [(1, 16, 64, 1), (257, 33, 97, 2), (3001, 128, 1024, 2), (3001, 128, 1024, 4), (1500, 20, 300, 3), (900, 66, 4096, 4),
                                     (2000, 9, 130, 1), (300, 12, 192, 4), (1200, 40, 20, 1)])
def test_screen_top_m(fg, monkeypatch, N, D, K, m):
    monkeypatch.setenv("GMM_SCREEN_MARKS", "1000")
    monkeypatch.setenv("GMM_SCREEN_PIECE", "768")
    X, pi, mu, var = _mixture(N, D, K, N + D + K, collapsed=3)
    X[N // 2] = 4000.0
    pi[K // 2] = 0.0
    if N == 300:
        pi[3:] = 0.0
    lj = np.asarray(orc.log_joint(X, pi, mu, var), np.float64)
    lz = np.logaddexp.reduce(lj, axis=1)
    want = np.sort(lj, axis=1)[:, ::-1][:, :m]
    with fg.Context(0) as c:
        idx, resp = (v.cpu().numpy() for v in c.gmm_assign_topm(_t(X), _t(pi), _t(mu), _t(var), m))
        idx2, resp2 = (v.cpu().numpy() for v in c.gmm_assign_topm(_t(X), _t(pi), _t(mu), _t(var), m))
        only = c.gmm_assign_topm(_t(X), _t(pi), _t(mu), _t(var), m, indices_only=True)
        only = (only[0] if isinstance(only, tuple) else only).cpu().numpy()
    assert np.array_equal(idx, idx2) and np.array_equal(resp, resp2) and np.array_equal(idx, only)
    assert idx.min() >= 0 and idx.max() < K and all(len(set(r)) == m for r in idx)
    got = np.take_along_axis(lj, idx.astype(np.int64), axis=1)
    near = np.abs(want) * 2e-6 + 1e-3
    ok = np.isneginf(want) if N == 300 else np.zeros_like(want, bool)
    assert np.all((got >= want - near) | (ok & np.isneginf(got)))
    with np.errstate(over="ignore"):
        r_ref = np.exp(got - lz[:, None])
    far = np.arange(N) == N // 2                            # (its log-densities of 1e7 leave fp32 little to tell)
    assert np.all(np.abs(resp - r_ref)[~far] <= 2e-4 * r_ref[~far] + 1e-6)


def test_screen_verdict_follows_the_whole_data(fg):
    """Rows in groups: a quarter of a tile whose posteriors are broad must not send sparse data to the dense kernels, wherever it lies, and a
    tenth of the data must, though the first tiles are sparse."""
    N, D, K = 60_000, 16, 256
    X, pi, mu, var = _mixture(N, D, K, 21)
    mu[K // 2:], var[K // 2:] = 12.0 + 0.05 * mu[K // 2:], 1.0
    rng = np.random.default_rng(4)
    X = (mu[rng.integers(0, K // 2, N)] + rng.normal(size=(N, D))).astype(np.float32)
    broad = (12.0 + rng.normal(size=(N // 10, D))).astype(np.float32)
    for first, n, sparse in [(0, 64, True), (256 * 100 + 30, 64, True), (N - 64, 64, True), (N - N // 10, N // 10, False)]:
        Y = X.copy()
        Y[first:first + n] = broad[:n]
        with fg.Context(0) as c:
            ref = orc.em_step(Y, pi, mu, var)
            got = c.gmm_em_step(_t(Y), _t(pi), _t(mu), _t(var))
            assert (c.gmm_last_exact_count() == K) == sparse, (first, n)
            assert abs(got[3] - ref[3]) <= 1e-5 * abs(ref[3])
            assert_stats_close(N, data_scale(Y), [v.cpu().numpy() for v in got[:3]], ref[:3], f"broad rows {first}+{n}")


def test_screen_forgets_earlier_calls(fg):
    """The same call gives the same bits whatever the context did before: sparse calls around broad ones of every entry point, and a fit whose
    posteriors sharpen on its way, twice."""
    N, D, K = 6000, 24, 128
    X, pi, mu, var = _mixture(N, D, K, 31)
    x, sparse = _t(X), [_t(a) for a in (pi, mu, var)]
    broad = [_t(pi), _t(X[:K]), _t(np.repeat(X.var(0)[None], K, 0))]
    offsets = np.array([0, N // 3, N], np.int64)

    def calls(c, params):
        out = list(c.gmm_em_step(x, *params)) + list(c.gmm_score_samples(x, *params)) + list(c.gmm_fisher_vectors(x, offsets, *params))
        out += list(c.gmm_assign_topm(x, *params, 2)) + list(c.gmm_kmeans_step(x, params[1])) + list(c.gmm_em_step_host(X, *[p.cpu().numpy() for p in params]))
        out.append(c.gmm_last_exact_count())
        return [v.cpu().numpy().copy() if torch.is_tensor(v) else np.array(v) for v in out]

    def fit(c):
        p = [v.clone() for v in broad]
        trace, _ = c.gmm_fit(x, *p, 12)
        return [trace] + [v.cpu().numpy() for v in p]

    with fg.Context(0) as c:
        first, fit1 = calls(c, sparse), fit(c)
        assert first[-1] == K
        for _ in range(2):
            calls(c, broad)
            assert all(np.array_equal(u, v) for u, v in zip(first, calls(c, sparse)))
        assert all(np.array_equal(u, v) for u, v in zip(fit1, fit(c)))


@pytest.mark.parametrize("N,D,K,screened", [(2000, 16, 64, False), (10_000, 32, 64, False), (10_000, 128, 1024, True)])
def test_screen_of_densities_only_where_it_is_faster(fg, N, D, K, screened):
    X, pi, mu, var = _mixture(N, D, K, 41)
    ref = np.logaddexp.reduce(np.asarray(orc.log_joint(X, pi, mu, var), np.float64), axis=1)
    with fg.Context(0) as c:
        logp, total = c.gmm_score_samples(_t(X), _t(pi), _t(mu), _t(var))
        assert c.gmm_last_path() == (fg.GMM_PATH_TENSOR if screened else fg.GMM_PATH_FP32)
    assert np.all(np.abs(logp.cpu().numpy() - ref) <= 1e-5 * np.abs(ref) + 1e-4) and abs(total - ref.sum()) <= 1e-5 * abs(ref.sum())


@pytest.mark.parametrize("N,D,K,m", [(2000, 16, 64, 1), (10_000, 32, 64, 1), (10_000, 100, 256, 2), (40_000, 32, 256, 2)])
def test_screen_of_assignments_where_the_rule_takes_either_way(fg, monkeypatch, N, D, K, m):
    # both sides of the rule on small calls: the same components, but for near ties, and the same responsibilities as by forced screening
    X, pi, mu, var = _mixture(N, D, K, 43)
    out = []
    for marks in (None, "1000"):
        if marks:
            monkeypatch.setenv("GMM_SCREEN_MARKS", marks)
        with fg.Context(0) as c:
            out.append([v.cpu().numpy() for v in c.gmm_assign_topm(_t(X), _t(pi), _t(mu), _t(var), m)])
    lj = np.asarray(orc.log_joint(X, pi, mu, var), np.float64)
    want = np.sort(lj, axis=1)[:, ::-1][:, :m]
    for idx, resp in out:
        got = np.take_along_axis(lj, idx.astype(np.int64), axis=1)
        weight = np.exp(want - np.logaddexp.reduce(lj, axis=1)[:, None]) > 1e-5     # (ranks without weight keep the order of a selection pass)
        assert np.all((got >= want - (np.abs(want) * 2e-6 + 1e-3))[weight])
    assert np.abs(out[0][1] - out[1][1]).max() <= 2e-4


@pytest.mark.parametrize("K", [128, 48])
@pytest.mark.parametrize("piece", [15, 5])
def test_screen_keeps_the_pieces_that_are_done(fg, monkeypatch, K, piece):
    """A region of broad posteriors that the look ahead does not meet, in the last or in a middle one of 16 pieces of 768 points: the pieces
    before it stay as they are, the dense kernels take the others, and every output is that of one pass over all points."""
    from oracle.kmeans import kmeans_step

    monkeypatch.setenv("GMM_SCREEN_MARKS", "10")
    monkeypatch.setenv("GMM_SCREEN_PIECE", "768")
    N, D = 16 * 768 + 100, 16
    _, pi, mu, var = _mixture(N, D, K, 51)
    mu[K // 2:], var[:] = 12.0 + 0.05 * mu[K // 2:], 1.0
    rng = np.random.default_rng(5)
    X = (mu[rng.integers(0, K // 2, N)] + rng.normal(size=(N, D))).astype(np.float32)
    first = piece * 768 + 450                              # (the rows that are looked at lie 384 into a piece)
    X[first:first + 300] = 12.0 + rng.normal(size=(300, D)).astype(np.float32)
    ref = orc.em_step(X, pi, mu, var)
    lj = np.asarray(orc.log_joint(X, pi, mu, var), np.float64)
    lz = np.logaddexp.reduce(lj, axis=1)
    a_r, _, _, inertia_r, gap = kmeans_step(X, mu.astype(np.float64))
    with fg.Context(0) as c:
        x, p = _t(X), [_t(pi), _t(mu), _t(var)]
        got = c.gmm_em_step(x, *p)
        assert c.gmm_last_exact_count() < K                # (the dense kernels had the last word)
        assert abs(got[3] - ref[3]) <= 1e-5 * abs(ref[3])
        assert_stats_close(N, data_scale(X), [v.cpu().numpy() for v in got[:3]], ref[:3], f"K={K} piece={piece}")
        q = [v.clone() for v in p]
        trace, done = c.gmm_fit(x, *q, 2)
        want = orc.fit(X, pi, mu, var, 2, var_floor=1e-6)["trace"]
        assert done == 2 and np.all(np.abs(trace - want) <= 1e-5 * np.abs(want))
        logp, total = c.gmm_score_samples(x, *p)
        assert np.all(np.abs(logp.cpu().numpy() - lz) <= 1e-5 * np.abs(lz) + 1e-4) and abs(total - lz.sum()) <= 1e-5 * abs(lz.sum())
        a, new, counts, inertia = c.gmm_kmeans_step(x, p[1])
        a = a.cpu().numpy()
        assert np.all((a == a_r) | (gap <= 1e-2)) and np.array_equal(counts.cpu().numpy(), np.bincount(a, minlength=K))
        assert abs(inertia - inertia_r) <= 1e-5 * inertia_r
        for k in np.unique(a)[:20]:
            np.testing.assert_allclose(new[k].cpu().numpy(), X[a == k].astype(np.float64).mean(0), rtol=0, atol=1e-4)
        for m in (1, 2):
            idx, resp = (v.cpu().numpy() for v in c.gmm_assign_topm(x, *p, m))
            at = np.take_along_axis(lj, idx.astype(np.int64), axis=1)
            assert np.all(at >= np.sort(lj, axis=1)[:, ::-1][:, :m] - 1e-3) and np.abs(resp - np.exp(at - lz[:, None])).max() <= 2e-4
        host = c.gmm_em_step_host(X, pi, mu, var)
        assert abs(host[3] - ref[3]) <= 1e-5 * abs(ref[3])
        assert_stats_close(N, data_scale(X), host[:3], ref[:3], "host")


@pytest.mark.parametrize("D,K", [(32, 64), (96, 48)])
@pytest.mark.parametrize("broad", [(0, 0), (0, 270_001), (150_000, 171_000), (255_000, 270_001), (70_000, 91_000)])
def test_host_streaming_takes_the_data_once_whatever_the_verdict(fg, D, K, broad):
    """Chunks of 8 MiB (5 of them, 13): sparse data, broad data, and a broad region in the second, a middle and the last chunk; each call gives the statistics of
    one pass, the same bits when repeated."""
    N = 270_001
    _, pi, mu, var = _mixture(100, D, K, 61)
    mu[K // 2:], var[:] = 0.02 * mu[K // 2:], 1.0
    rng = np.random.default_rng(6)
    X = rng.normal(size=(N, D)).astype(np.float32)
    X += mu[rng.integers(0, K // 2, N)]
    X[broad[0]:broad[1]] = rng.normal(size=(broad[1] - broad[0], D)).astype(np.float32)
    ref = orc.em_step(X, pi, mu, var)
    with fg.Context(0) as c:
        out = [c.gmm_em_step_host(X, pi, mu, var) for _ in range(2)]
        assert (c.gmm_last_exact_count() == K) == (broad[1] == 0)
    for u, v in zip(*out):
        assert np.array_equal(u, v)
    assert abs(out[0][3] - ref[3]) <= 1e-5 * abs(ref[3])
    assert_stats_close(N, data_scale(X), out[0][:3], ref[:3], f"K={K} broad={broad}")


@pytest.mark.parametrize("D,K,N,left", [(128, 1024, 3000, 770), (96, 48, 200_000, 770)])
def test_screen_does_without_where_memory_is_short(fg, D, K, N, left):
    """Room (in MiB) for what the dense kernels need (at most 590), not for the planes and lists on top (816 in all at 128 x 1024, 783 at 96 x 48): the call runs, as it does without a screening path, and the next
    shape is screened again when there is room."""
    X, pi, mu, var = _mixture(N, D, K, 71)
    ref = orc.em_step(X, pi, mu, var)
    args = [_t(a) for a in (X, pi, mu, var)]
    small = [_t(a) for a in _mixture(2000, 16, 64, 72)]
    with fg.Context(0) as c:
        c.gmm_em_step(*small)                              # (what the first calls allocate besides)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        hog = torch.empty(torch.cuda.mem_get_info()[0] - (left << 20) + int(fg.lib.gmm_scratch_bytes(16, 64)), dtype=torch.uint8, device=DEV)
        launches = []
        for _ in range(2):
            before = c.gmm_launch_count()
            got = c.gmm_em_step(*args)
            launches.append(c.gmm_launch_count() - before)
            assert abs(got[3] - ref[3]) <= 1e-5 * abs(ref[3])
            assert_stats_close(N, data_scale(X), [v.cpu().numpy() for v in got[:3]], ref[:3], "short of memory")
        del hog, got
        torch.cuda.empty_cache()
        c.gmm_em_step(*small)
        assert c.gmm_last_exact_count() == 64
        before = c.gmm_launch_count()
        c.gmm_em_step(*args)
        assert c.gmm_last_exact_count() == K and launches[0] == launches[1] != c.gmm_launch_count() - before


def test_screen_of_large_groups_of_which_the_last_is_broad(fg):
    """Fisher vectors of four groups that are larger than one CTA sorts; a broad region that the look ahead does not meet sends the call to the dense
    kernels when three of them are done."""
    from oracle.fisher import fisher_vectors

    N, D, K = 160_000, 16, 64
    _, pi, mu, var = _mixture(100, D, K, 81)
    mu[K // 2:], var[:], pi[:] = 0.02 * mu[K // 2:], 1.0, 1.0 / K
    rng = np.random.default_rng(8)
    X = (mu[rng.integers(0, K // 2, N)] + rng.normal(size=(N, D))).astype(np.float32)
    X[-3000:-500] = rng.normal(size=(2500, D)).astype(np.float32)
    offsets = np.arange(5, dtype=np.int64) * 40_000
    ref = fisher_vectors(X, offsets, pi, mu, var)
    lz = orc.responsibilities(X, pi, mu, var)[1]
    with fg.Context(0) as c:
        G, ll = c.gmm_fisher_vectors(_t(X), offsets, _t(pi), _t(mu), _t(var))
    assert abs(ll - lz.sum()) <= 1e-5 * abs(lz.sum())
    # (the dense kernels' bound of flashgmm.h, A_k = N_k / (T sqrt(pi_k)) <= 1/4 here)
    assert np.abs(G.cpu().numpy() - ref).max() <= 2e-5 * (1 + np.abs(ref).max()) + 0.25 * (1e-3 + 4e-5 * (1 + float((mu * mu).max())))
