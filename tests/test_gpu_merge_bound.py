"""The merge step's bound (a pair is refused without factorising its matrix) against the
oracle, which evaluates every pair: mixtures whose clusters lie from on top of one another to
far apart, with few and with many points, so that pairs are refused, left open and merged in
one sweep; the split/merge decisions, counters and labels must be the oracle's, sweep by sweep."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,K,N,spread", [(1, 9, 300, 2.0), (2, 24, 4_000, 1.5), (3, 12, 150, 0.3), (9, 33, 2_000, 0.8),
                                          (33, 6, 500, 0.1), (40, 20, 6_000, 0.25)])
def test_merge_decisions_match_oracle(d, K, N, spread):
    import __graft_entry__

    __graft_entry__.build()
    import oracle as O
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(10 * d + K)
    mu = rng.standard_normal((K, d)) * spread
    scale = np.exp(rng.uniform(-1, 1, K))
    y = rng.choice(K, N, p=rng.dirichlet(np.full(K, 0.7))).astype(np.int32)
    X = mu[y] + scale[y, None] * rng.standard_normal((N, d)) + 100.0  # data need not be centred
    prior = dict(kappa0=0.5, m0=np.full(d, 99.0), nu0=d + 2.5, psi0=np.eye(d) * 1.5)
    o = O.Oracle(O.NIW, d, 64, 2.0, burn_out=2, **prior)
    g = P.DPMM(P.PRIOR_NIW, d, 64, 2.0, prec=P.PREC_FP64_PLAIN, burn_out=2, **prior)
    y = np.unique(y, return_inverse=True)[1].astype(np.int32)
    zb = rng.integers(0, 2, N).astype(np.uint8)
    for c in (o, g):
        c.set_data(X)
        c.set_state(int(y.max()) + 1, y, zb)
    merges = 0
    for t in range(6):
        o.sweep(1, 77)
        g.sweep(1, 77)
        co, cg = o.counters(), g.counters()
        assert dict(co) == dict(cg), t
        zo, zbo = o.labels()
        zg, zbg = g.labels()
        assert o.K == g.K and np.array_equal(zo, zg) and np.array_equal(zbo, zbg), t
        merges += cg["merges"]
    if spread < 1.0:
        assert merges > 0  # the case does reach the pairs that the bound leaves open
    g.close()
