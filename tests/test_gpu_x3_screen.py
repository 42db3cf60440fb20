"""The screened label step of large BF16X3 data against the three products for every point:
the same labels where nearly every point is decided by one product, where clusters overlap so
that more points stay open than the gathered tiles hold (all are scored then, also in the
sweeps that follow without a screening), with ragged sizes, weights of zero, and d on either
side of 64.  The full step is run through label_scores' kernel and the same Gumbel values."""
import numpy as np
import pytest

from test_gpu_labels_niw import _uniforms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,K,N,spread", [(128, 6, 70_001, 4.0), (100, 9, 65_537, 0.6), (128, 5, 66_000, 0.0),
                                          (64, 7, 262_145, 3.0), (40, 12, 300_000, 0.8)])
def test_screened_labels_are_those_of_three_products(d, K, N, spread):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(d + K)
    mu = rng.standard_normal((K, d)) * spread
    y = rng.integers(0, K, N)
    X = (mu[y] + rng.standard_normal((N, d))).astype(np.float32)
    W = np.triu(rng.standard_normal((3 * K, d, d)) * 0.3 / np.sqrt(d), 1) + np.eye(d) * rng.uniform(0.7, 1.4, (3 * K, d, 1))
    ldw = np.log(np.diagonal(W, axis1=1, axis2=2)).sum(1)
    logw = np.log(rng.dirichlet(np.ones(K), 3).T.reshape(-1))
    logw[3] = -np.inf
    mus = np.repeat(mu, 3, 0) + 0.01 * rng.standard_normal((3 * K, d))
    g = P.DPMM(P.PRIOR_NIW, d, 16, 1.0, prec=P.PREC_BF16X3, psi0=np.eye(d))
    g.set_data(X)
    g.set_state(K, (np.arange(N) % K).astype(np.int32), np.zeros(N, np.uint8))
    g.set_params(K, dict(logw=logw, mu=mus, W=W, logdetW=ldw))
    v = g.label_scores() + _uniforms(N, K, 99, False)
    want = v.argmax(1)
    live = np.unique(want)
    top = np.sort(v, 1)
    sure = top[:, -1] - top[:, -2] > 1e-3 * np.maximum(1.0, np.abs(top[:, -1]))  # FP32 sums and logarithms
    g.set_mask(2)
    for _ in range(3):  # the same sweep index each time
        g.set_params(K, dict(logw=logw, mu=mus, W=W, logdetW=ldw))
        g.set_iter(0)
        g.sweep(1, 99)
        z, _ = g.labels()
        assert sure.mean() > 0.9
        assert np.array_equal(z[sure], np.searchsorted(live, want)[sure])
    g.close()
