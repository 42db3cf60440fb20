"""The pruned Gaussian label step on the CUDA cores, against Gumbel-max over every cluster's
score: odd and even dimensions, more contenders than a thread holds, more clusters than the
data have, clusters of weight zero, one cluster, and points that come in no order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _uniforms(N, K, seed, prec64):
    """Gumbel values of tag Z from the oracle-independent Philox of the header's layout."""
    def mul(a, b):
        p = np.uint64(a) * b.astype(np.uint64)
        return (p >> np.uint64(32)).astype(np.uint32), p.astype(np.uint32)

    out = np.empty((N, K))
    i = np.arange(N, dtype=np.uint32)
    for blk in range((K + 1) // 2):
        c = [i.copy(), np.zeros(N, np.uint32), np.full(N, (5 << 24) | blk, np.uint32), np.zeros(N, np.uint32)]
        k0, k1 = seed & 0xFFFFFFFF, seed >> 32
        for _ in range(10):
            h0, l0 = mul(0xD2511F53, c[0])
            h1, l1 = mul(0xCD9E8D57, c[2])
            c = [h1 ^ c[1] ^ np.uint32(k0), l1, h0 ^ c[3] ^ np.uint32(k1), l0]
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        for h in range(2):
            if 2 * blk + h >= K:
                continue
            a, b = c[2 * h].astype(np.uint64), c[2 * h + 1].astype(np.uint64)
            if prec64:
                u = (2 * (((a >> np.uint64(6)) << np.uint64(26)) | (b >> np.uint64(6))) + 1).astype(np.float64) * 2.0 ** -53
            else:
                u = (2 * (a >> np.uint64(9)) + 1).astype(np.float64) * 2.0 ** -24
            out[:, 2 * blk + h] = -np.log(-np.log(u))
    return out


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("d,K,N,spread", [(1, 3, 33, 1.0), (2, 40, 5_000, 0.5), (3, 1, 100, 1.0), (7, 19, 3_001, 0.3),
                                          (8, 64, 4_097, 2.0), (31, 5, 777, 3.0), (32, 20, 20_001, 4.0), (33, 12, 1_000, 0.05)])
def test_labels_are_those_of_every_score(prec, d, K, N, spread):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(d * 1000 + K)
    mu = rng.standard_normal((3 * K, d)) * spread
    y = rng.integers(0, K, N)
    X = mu[3 * y] + rng.standard_normal((N, d))
    dt = np.float64 if prec == "fp64" else np.float32
    X = X.astype(dt)
    W = np.triu(rng.standard_normal((3 * K, d, d)) * 0.2, 1) + np.eye(d) * rng.uniform(0.5, 1.5, (3 * K, d, 1))
    ldw = np.log(np.diagonal(W, axis1=1, axis2=2)).sum(1)
    logw = np.log(rng.dirichlet(np.ones(K), 3).T.reshape(-1))
    if K > 4:
        logw[3 * 2] = -np.inf  # a cluster of weight zero
    g = P.DPMM(P.PRIOR_NIW, d, max(K, 2), 1.0, prec=P.PREC_FP64_PLAIN if prec == "fp64" else P.PREC_FP32, psi0=np.eye(d))
    g.set_data(X)
    start = rng.integers(0, K, N).astype(np.int32)
    start[:K] = np.arange(min(K, N))[:K] if N >= K else start[:K]
    g.set_state(K, start, np.zeros(N, np.uint8))
    g.set_params(K, dict(logw=logw, mu=mu, W=W, logdetW=ldw))
    scores = g.label_scores()  # every cluster in full, by the step's own precision
    g.set_mask(2)
    g.sweep(1, 99)
    # labels as drawn: emptied clusters are removed afterwards, their ids closed up in order
    z, _ = g.labels()
    v = scores + _uniforms(N, K, 99, prec == "fp64")
    want = v.argmax(1)
    live = np.unique(want)
    top = np.sort(v, 1)
    # the GPU's logarithms and the last rounding of s + G against numpy's
    tol = 1e-9 if prec == "fp64" else 1e-4 * np.maximum(1.0, np.abs(top[:, -1]))
    sure = np.ones(N, bool) if K == 1 else (top[:, -1] - top[:, -2] > tol)
    assert sure.mean() > 0.99
    assert np.array_equal(z[sure], np.searchsorted(live, want)[sure])
    g.close()
