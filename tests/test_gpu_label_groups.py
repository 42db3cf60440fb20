"""The TF32 label step where one group of clusters holds K_max (nothing is carried over groups),
where K fills one group of several, and over several groups: the labels are the argmax of the
step's own scores and the same Gumbel values, for clusters that overlap."""
import numpy as np
import pytest

from test_gpu_labels_niw import _uniforms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,K,K_max", [(8, 12, 64), (9, 40, 64), (32, 12, 16), (32, 26, 64), (32, 27, 64), (32, 60, 64)])
def test_labels_are_the_argmax_of_their_scores(d, K, K_max):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    N = 20_001
    rng = np.random.default_rng(d + K)
    mu = 0.5 * rng.standard_normal((K, d))
    X = (mu[rng.integers(0, K, N)] + rng.standard_normal((N, d))).astype(np.float32)
    params = dict(logw=np.log(np.full(3 * K, 1.0 / K)), mu=np.repeat(mu, 3, 0), W=np.tile(np.eye(d), (3 * K, 1, 1)),
                  logdetW=np.zeros(3 * K))
    g = P.DPMM(P.PRIOR_NIW, d, K_max, 1.0, prec=P.PREC_TF32, psi0=np.eye(d))
    g.set_data(X)
    g.set_state(K, (np.arange(N) % K).astype(np.int32), np.zeros(N, np.uint8))
    g.set_params(K, params)
    v = g.label_scores() + _uniforms(N, K, 99, False)
    want = v.argmax(1)
    live = np.unique(want)
    top = np.sort(v, 1)
    sure = top[:, -1] - top[:, -2] > 1e-3  # scores below 128 and Gumbel values in FP32: three roundings of 8e-6
    g.set_mask(2)
    g.set_iter(0)
    g.sweep(1, 99)
    z, _ = g.labels()
    g.close()
    assert sure.mean() > 0.9 and np.array_equal(z[sure], np.searchsorted(live, want)[sure])
