"""Label steps without the parameter step where K exceeds the clusters whose parameters were last drawn or set
(after a split, or a state of more clusters): the clusters beyond keep the parameters they had, and the
labels and sub-labels are those of their FP64 scores, as label_scores gives them."""
import numpy as np
import pytest

from test_gpu_labels_niw import _uniforms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,N", [(2, 500), (8, 500), (9, 700), (32, 900), (40, 300)])
def test_clusters_beyond_the_last_draw(d, N):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(d)
    K = 4
    mu = np.stack([np.full(d, v) for v in (0.0, 3.0, 30.0, 33.0)])
    X = mu[rng.integers(0, K, N)] + rng.standard_normal((N, d)) * 0.7 + rng.uniform(-1, 1, (N, 1))

    def params(means):
        k = len(means)
        sub = np.repeat(means, 3, 0)  # sub-clusters 80 apart in the first coordinate
        sub[1::3, 0] -= 40.0
        sub[2::3, 0] += 40.0
        return dict(logw=np.log(np.tile([1 / K, 0.5, 0.5], k)), mu=sub, W=np.repeat(np.eye(d)[None], 3 * k, 0), logdetW=np.zeros(3 * k))

    g = P.DPMM(P.PRIOR_NIW, d, 8, 1.0, prec=P.PREC_FP64_PLAIN, psi0=np.eye(d))
    g.set_data(X)
    state = ((np.arange(N) % K).astype(np.int32), np.zeros(N, np.uint8))
    g.set_state(K, *state)
    g.set_params(K, params(mu))
    g.set_params(2, params(mu[:2] + 50.0))  # clusters 0 and 1 move; 2 and 3 keep their parameters
    g.set_state(K, *state)
    v = g.label_scores() + _uniforms(N, K, 99, True)
    g.set_mask(2)
    g.sweep(1, 99)
    z, zb = g.labels()
    g.close()
    want = v.argmax(1)
    assert np.array_equal(z, np.searchsorted(np.unique(want), want))
    off = X[:, 0] - mu[want, 0] - np.where(want < 2, 50.0, 0.0)
    sure = np.abs(80 * off) > 41  # the scores' difference against the Gumbels'
    assert sure.mean() > 0.3 and np.array_equal(zb[sure], off[sure] > 0)
