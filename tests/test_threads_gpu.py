"""Contexts of several threads, each on its own stream, at work on different shapes at the same time."""
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _calls(fg, K, D, path, rounds, failures):
    """Every entry point whose kernels take shared memory by shape; the same bits in every round."""
    stream = torch.cuda.Stream()
    try:
        with torch.cuda.stream(stream), fg.Context(0) as c:
            g = torch.Generator(device=DEV)
            g.manual_seed(K)
            mu = torch.randn((K, D), device=DEV, generator=g) * 3
            X = mu[torch.randint(0, K, (3000,), device=DEV, generator=g)] + torch.randn((3000, D), device=DEV, generator=g)
            var, pi = torch.ones((K, D), device=DEV), torch.full((K,), 1 / K, device=DEV)
            groups = np.array([0, 700, 3000], np.int64)
            c.gmm_set_path(path)
            first = None
            for _ in range(rounds):
                out = list(c.gmm_em_step(X, pi, mu, var))
                idx, resp = c.gmm_assign_topm(X, pi, mu, var, 2)
                out += [idx, resp, c.gmm_build_posting_lists(idx, resp, K)[0], c.gmm_fisher_vectors(X, groups, pi, mu, var)[0]]
                out += list(c.gmm_kmeans_step(X, mu))
                out = [v.cpu() if torch.is_tensor(v) else v for v in out]
                first = first or out
                assert all(torch.equal(u, v) if torch.is_tensor(u) else u == v for u, v in zip(first, out))
    except Exception as e:      # (a thread's exception is the test's)
        failures.append(f"K={K} D={D} path={path}: {e}")


def test_contexts_on_several_threads_take_different_shapes():
    from paper_2606_10896_b200 import flashgmm as fg

    failures = []
    shapes = [(4096, 16, fg.GMM_PATH_AUTO), (64, 16, fg.GMM_PATH_AUTO), (64, 128, fg.GMM_PATH_FP32), (40, 100, fg.GMM_PATH_FP32)]
    threads = [threading.Thread(target=_calls, args=(fg, K, D, path, 60, failures)) for K, D, path in shapes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures


def _unclean(fg, k, D, K, start, failures):
    """Steps on data with an infinity in every tile of 256 points, in turn with clean data; the same bits in every round."""
    stream = torch.cuda.Stream()
    try:
        with torch.cuda.stream(stream), fg.Context(0) as c:
            g = torch.Generator(device=DEV)
            g.manual_seed(k)
            mu = torch.randn((K, D), device=DEV, generator=g) * 3
            X = mu[torch.randint(0, K, (60_000,), device=DEV, generator=g)] + torch.randn((60_000, D), device=DEV, generator=g)
            var, pi = torch.ones((K, D), device=DEV), torch.full((K,), 1 / K, device=DEV)
            bad = X.clone()
            bad[k::256, D - 1] = float("inf")
            first = None
            start.wait()
            for _ in range(25):
                for call in (lambda: c.gmm_kmeans_step(bad, mu), lambda: (c.gmm_assign_topm(bad, pi, mu, var, 2), c.gmm_sync_status())):
                    with pytest.raises(fg.GmmError) as e:
                        call()
                    assert e.value.code == fg.GMM_ENUMERIC
                out = list(c.gmm_kmeans_step(X, mu)) + list(c.gmm_em_step(X, pi, mu, var))
                assert c.gmm_last_exact_count() == K
                out = [v.cpu().numpy() if torch.is_tensor(v) else np.asarray(v) for v in out]
                first = first or out
                assert all(np.array_equal(u, v, equal_nan=True) for u, v in zip(first, out))
    except Exception as e:      # (a thread's exception is the test's)
        failures.append(f"K={K} D={D}: {e}")


# The screening sweep finds values that are not finite while it runs, and CTAs that start later than that (beside another context's kernels
# they do) leave as a whole or take part as a whole.
def test_contexts_on_several_threads_meet_values_that_are_not_finite():
    from paper_2606_10896_b200 import flashgmm as fg

    failures = []
    shapes = [(40, 64), (96, 300), (128, 64), (16, 200)]
    start = threading.Barrier(len(shapes))
    threads = [threading.Thread(target=_unclean, args=(fg, k, D, K, start, failures)) for k, (D, K) in enumerate(shapes)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
