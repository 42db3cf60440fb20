"""New data under the parameters last set (the parameter step masked out) with BF16X3: a fitted
model labels another batch through update_data, stage_data or a second set_data, also where the
first data were too few for the screened label step.  The labels are those of label_scores (the
three products for every point) and the same Gumbel values.  Standard deviations run from 1 to
0.01 and means lie about 40 apart, in pairs, so far that few
points lie between two clusters, and that a product of x_h and W_h alone still picks the wrong
cluster of a pair for some."""
import numpy as np
import pytest

from test_gpu_labels_niw import _uniforms

pytestmark = pytest.mark.gpu
K = 16


# with mask 6 (merges too) not set_data: a new state's first FP32 statistics are not about the clusters' means
@pytest.mark.parametrize("how,d,N,apart,mask", [(how, *size, 2) for how in ("update_data", "stage_data", "set_data")
                                                for size in ((128, 70_001, 1.1), (64, 262_145, 1.7))] +
                         [("update_data", 64, 262_145, 1.7, 6), ("stage_data", 64, 262_145, 1.7, 6)])
def test_labels_of_new_data(how, d, N, apart, mask):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(d)
    Q = np.linalg.qr(rng.standard_normal((d, d)))[0]
    L = np.linalg.cholesky(Q @ np.diag(np.geomspace(1, 0.01, d) ** 2) @ Q.T)
    mu = np.repeat(40 * rng.standard_normal((K // 2, d)), 2, 0)
    mu[1::2] += apart * rng.standard_normal((K // 2, d)) @ L.T
    X, old = ((mu[rng.integers(0, K, N)] + rng.standard_normal((N, d)) @ L.T).astype(np.float32) for _ in range(2))
    if how == "set_data":  # too few points to be screened, with the same centre
        old = (old[:4_000] - old[:4_000].mean(0, dtype=np.float64) + X.mean(0, dtype=np.float64)).astype(np.float32)
    W = np.repeat(np.linalg.inv(L).T[None], 3 * K, 0)
    params = dict(logw=np.log(np.tile([1 / K, 0.5, 0.5], K)), mu=np.repeat(mu, 3, 0), W=W,
                  logdetW=np.log(np.diagonal(W, axis1=1, axis2=2)).sum(1))
    g = P.DPMM(P.PRIOR_NIW, d, 16, 1.0, prec=P.PREC_BF16X3, psi0=np.eye(d) * 1e-6)

    def settle(n):
        g.set_state(K, (np.arange(n) % K).astype(np.int32), np.zeros(n, np.uint8))

    g.set_data(old)
    settle(len(old))
    g.set_params(K, params)
    g.set_mask(mask)
    getattr(g, how)(X)
    if how == "set_data":
        settle(N)
    g.sweep(1, 99)
    z, _ = g.labels()
    assert g.K == K
    v = g.label_scores() + _uniforms(N, K, 99, False)
    g.close()
    top = np.sort(v, 1)
    sure = top[:, -1] - top[:, -2] > 1e-3 * np.maximum(1.0, np.abs(top[:, -1]))  # FP32 sums and logarithms
    assert sure.mean() > 0.9
    assert np.array_equal(z[sure], v.argmax(1)[sure])
