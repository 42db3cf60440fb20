"""FP64 labels of points whose whitened distances leave FP32's range (a sentinel, an outlier, units far
from 1): the label is that of the FP64 scores and Gumbel values, which are finite."""
import numpy as np
import pytest

from test_gpu_labels_niw import _uniforms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-2, 1e-10, 1e-25, 1e-45, 1e30])
@pytest.mark.parametrize("d,K,N", [(9, 5, 400), (12, 20, 333), (32, 12, 1_000)])
def test_far_points(d, K, N, scale):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(d)
    mu = 3.0 * rng.standard_normal((K, d)) * scale
    X = mu[rng.integers(0, K, N)] + rng.standard_normal((N, d)) * scale
    for i, far in enumerate([1e18, 1.9e19, 1e20, 1e25, 1e30, 4e38, 1e45, -1e20, -1e39]):
        X[3 * i + 1] = far * scale  # every feature
        X[3 * i + 2, i % d] = far * scale  # one
    W = (np.triu(rng.standard_normal((K, d, d)) * 0.2, 1) + np.eye(d) * rng.uniform(0.5, 1.5, (K, d, 1))) / scale
    logw = np.log(np.repeat(rng.dirichlet(np.ones(K)), 3))
    logw[3] = -np.inf
    ldw = np.log(np.diagonal(W, axis1=1, axis2=2)).sum(1)
    g = P.DPMM(P.PRIOR_NIW, d, K, 1.0, prec=P.PREC_FP64_PLAIN, psi0=np.eye(d) * scale * scale)
    g.set_data(X)
    g.set_state(K, (np.arange(N) % K).astype(np.int32), np.zeros(N, np.uint8))
    g.set_params(K, dict(logw=logw, mu=np.repeat(mu, 3, 0), W=np.repeat(W, 3, 0), logdetW=np.repeat(ldw, 3)))
    v = g.label_scores() + _uniforms(N, K, 99, True)
    g.set_mask(2)
    g.sweep(1, 99)
    z, _ = g.labels()
    g.close()
    want = v.argmax(1)
    top = np.sort(v, 1)
    sure = top[:, -1] - top[:, -2] > 1e-9 * np.maximum(1.0, np.abs(top[:, -1]))
    assert np.isfinite(np.delete(v, 1, 1)).all() and sure.mean() > 0.98
    live = np.unique(want)
    assert np.array_equal(z[sure], np.searchsorted(live, want)[sure])


@pytest.mark.parametrize("d,K,N", [(2, 4, 501), (8, 3, 700), (12, 5, 999), (33, 4, 300)])
def test_gumbels_lost_in_large_scores(d, K, N):
    """Scores so large that s + G rounds to s: equal clusters and equal sub-clusters are ties, which go to the
    lower index, as with every FP64 value drawn; and scores near 1e13, where the sums' grid is 0.002."""
    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(d)
    mu = np.repeat(rng.standard_normal((K, d)), 2, 0)  # pairs of equal clusters
    W = np.repeat(np.triu(rng.standard_normal((K, d, d)) * 0.2, 1) + np.eye(d) * rng.uniform(0.5, 1.5, (K, d, 1)), 2, 0)
    ldw = np.log(np.diagonal(W, axis1=1, axis2=2)).sum(1)
    far = rng.choice([4e6, 1e12], N)
    X = rng.standard_normal((N, d))
    X *= (far / np.linalg.norm(X, axis=1))[:, None]
    logw = np.log(np.tile([1 / (2 * K), 0.5, 0.5], 2 * K))
    g = P.DPMM(P.PRIOR_NIW, d, 2 * K, 1.0, prec=P.PREC_FP64_PLAIN, psi0=np.eye(d))
    g.set_data(X)
    g.set_state(2 * K, (np.arange(N) % (2 * K)).astype(np.int32), np.ones(N, np.uint8))
    g.set_params(2 * K, dict(logw=logw, mu=np.repeat(mu, 3, 0), W=np.repeat(W, 3, 0), logdetW=np.repeat(ldw, 3)))
    s = g.label_scores()
    v = s + _uniforms(N, 2 * K, 99, True)
    g.set_mask(2)
    g.sweep(1, 99)
    z, zb = g.labels()
    g.close()
    want = v.argmax(1)
    assert np.array_equal(z, np.searchsorted(np.unique(want), want))
    lost = far > 1e11
    assert (want[lost] % 2 == 0).all() and not zb[lost].any() and zb[~lost].any()
