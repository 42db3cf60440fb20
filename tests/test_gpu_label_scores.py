"""label_scores before any parameters exist: the tensor-core paths refuse it, and the chain goes on as if it had
not been called, also when K grows beyond the value it had then."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["TF32", "BF16", "BF16X3", "FP32", "FP64_PLAIN"])
def test_the_chain_goes_on(prec):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(5)
    N, d, K = 3_000, 16, 6
    if prec == "BF16":
        theta = rng.dirichlet(np.full(d, 0.1), K)
        X = np.stack([rng.multinomial(60, theta[i % K]) for i in range(N)]).astype(np.int32)
    else:
        X = (6.0 * rng.standard_normal((K, d))[np.arange(N) % K] + rng.standard_normal((N, d))).astype(np.float32)
    z0, zb0 = np.zeros(N, np.int32), (np.arange(N) % K < 3).astype(np.uint8)

    def chain(ask):
        g = P.DPMM(P.PRIOR_DIRICHLET if prec == "BF16" else P.PRIOR_NIW, d, 16, 10.0, prec=getattr(P, "PREC_" + prec), burn_out=1)
        g.set_data(X)
        g.set_state(1, z0, zb0)
        if ask and prec in ("TF32", "BF16"):
            with pytest.raises(P.DPMMError):
                g.label_scores()
        elif ask:
            g.label_scores()
        out = []
        for _ in range(6):
            g.sweep(1, 3)
            out.append((g.K, *g.labels()))
        scores = g.label_scores()
        g.close()
        return out, scores

    (a, sa), (b, sb) = chain(False), chain(True)
    assert a[-1][0] > 1 and np.array_equal(sa, sb)
    for u, v in zip(a, b):
        assert u[0] == v[0] and np.array_equal(u[1], v[1]) and np.array_equal(u[2], v[2])
