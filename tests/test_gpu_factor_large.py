"""The parameter draws in FP64 at large dimensions: W in shared memory beside the
factor (d <= 153) and in global memory (154 to 160).  W solves U^T W = B and mu is m_n + W^-T eps /
sqrt(kappa_n), where B and eps hang on the seed, the slot and the counts alone: B = U^T W and eps, formed in
numpy from the draws of two data sets with the same counts, are the same.  Values are small whole
numbers whose mean is 0, so that the FP32 statistics are exact; N = 40 d keeps the factors'
condition below 100, so d^2 roundings of 2^-53 are below 3e-10 of the largest entry."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [128, 153, 154, 155, 158, 160])
def test_draws_are_the_same_variates(d):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(d)
    h = 20 * d
    half = rng.integers(-4, 5, (h, d)) + rng.integers(-2, 3, d)
    z = np.repeat(np.arange(2, dtype=np.int32), h)
    zb = np.tile(np.arange(h) % 2, 2).astype(np.uint8)
    found = []
    for mixed in (False, True):
        A = half + np.roll(half, 1, 1) if mixed else half
        X = np.concatenate([A, -A]).astype(np.float32)
        g = P.DPMM(P.PRIOR_NIW, d, 4, 2.0, prec=P.PREC_FP32, kappa0=1.0, m0=np.zeros(d), nu0=d + 3.0, psi0=np.eye(d))
        g.set_data(X)
        g.set_state(2, z, zb)
        g.set_iter(3)
        g.set_mask(1)
        g.sweep(1, 99)
        p = g.params()
        g.close()
        for s in range(6):
            k, sub = s // 3, s % 3 - 1
            Y = X[(z == k) & ((zb == sub) | (sub < 0))].astype(np.float64)
            n, m = len(Y), Y.mean(0)
            U = np.linalg.cholesky(np.eye(d) + (Y - m).T @ (Y - m) + n / (1 + n) * np.outer(m, m))
            B = U.T @ p["W"][s]
            assert np.abs(np.tril(p["W"][s], -1)).max() == 0 and (np.diagonal(B) > 0).all()
            assert abs(p["logdetW"][s] - np.log(np.diagonal(p["W"][s])).sum()) <= 1e-9 * d
            eps = p["W"][s].T @ (p["mu"][s] - n * m / (1 + n)) * np.sqrt(1 + n)
            found.append((B, eps))
    for (B, eps), (C, eta) in zip(found[:6], found[6:]):
        assert np.abs(B - C).max() <= 1e-9 * np.abs(B).max() and np.abs(eps - eta).max() <= 1e-9 * np.abs(eps).max() + 1e-8
        up = B[np.triu_indices(d, 1)]
        assert abs(up.mean()) < 0.1 and abs(up.std() - 1) < 0.1 and np.abs(np.tril(B, -1)).max() <= 1e-9 * np.abs(B).max()
