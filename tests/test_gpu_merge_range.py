"""The merge bounds where a feature's scatter is a denormal number in FP32: one feature in units so small
that its summed squares are near 2e-45, all others of unit scale, in which clusters differ by that
feature alone.  The decisions are the oracle's, which evaluates every pair in FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,K,n,seed", [(24, 26, 4_000, 0), (24, 26, 4_000, 3), (1, 26, 300, 1)])
def test_decisions_at_denormal_scatter(d, K, n, seed):
    import __graft_entry__

    __graft_entry__.build()
    import oracle as O
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(seed)
    scale = np.ones(d)
    scale[0] = np.sqrt(1.45 * 1.4013e-45 / n)  # n squares: 1.45 of the least denormal, which rounds to 1
    mu = np.zeros((K, d))
    mu[:, 0] = rng.uniform(0, 4, K) * scale[0]
    y = (np.arange(K * n) % K).astype(np.int32)
    X = mu[y] + rng.standard_normal((K * n, d)) * scale
    zb = rng.integers(0, 2, K * n).astype(np.uint8)
    prior = dict(kappa0=1.0, m0=np.zeros(d), nu0=d + 3.0, psi0=np.diag(scale ** 2))
    o = O.Oracle(O.NIW, d, 64, 2.0, burn_out=15, **prior)
    g = P.DPMM(P.PRIOR_NIW, d, 64, 2.0, prec=P.PREC_FP64_PLAIN, burn_out=15, **prior)
    for c in (o, g):
        c.set_data(X)
        c.set_state(K, y, zb)
    o.sweep(1, 77, mask=O.MASK_SPLITMERGE)
    g.set_mask(4)
    g.sweep(1, 77)
    assert o.counters()["merges"] > 0
    assert dict(o.counters()) == dict(g.counters())
    zo, _ = o.labels()
    zg, _ = g.labels()
    g.close()
    assert o.K == len(np.unique(zg)) and np.array_equal(zo, zg)
