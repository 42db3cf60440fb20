"""Merge decisions under the bounds, in every way that they are taken, against the oracle, which evaluates
every pair: within the merge kernel (d < 76, more than two slots and pairs an SM) and by a kernel
ahead of it (more than one an SM).  Clusters overlap, so that pairs are refused, left open and merged."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,K,N,spread", [(33, 30, 3_000, 0.1), (40, 30, 6_000, 0.25), (75, 26, 4_000, 0.15),
                                          (80, 24, 4_000, 0.15), (128, 24, 5_000, 0.12), (100, 40, 2_000, 0.3)])
def test_bounded_merge_decisions(d, K, N, spread):
    import torch

    import __graft_entry__

    __graft_entry__.build()
    import oracle as O
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(10 * d + K)
    mu = rng.standard_normal((K, d)) * spread * rng.choice([0.2, 1.0, 4.0], (K, 1))
    scale = np.exp(rng.uniform(-0.5, 0.5, K))
    y = np.concatenate([np.arange(K), rng.choice(K, N - K, p=rng.dirichlet(np.full(K, 2.0)))]).astype(np.int32)
    X = mu[y] + scale[y, None] * rng.standard_normal((N, d)) + 100.0
    zb = rng.integers(0, 2, N).astype(np.uint8)
    prior = dict(kappa0=0.5, m0=np.full(d, 99.0), nu0=d + 2.5, psi0=np.eye(d) * 1.5)
    o = O.Oracle(O.NIW, d, 64, 2.0, burn_out=15, **prior)
    g = P.DPMM(P.PRIOR_NIW, d, 64, 2.0, prec=P.PREC_FP64_PLAIN, burn_out=15, **prior)
    for c in (o, g):
        c.set_data(X)
        c.set_state(K, y, zb)
    g.set_mask(4)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    merges = 0
    for t in range(4):
        items = 3 * o.K + o.K * (o.K - 1) // 2
        assert t > 0 or items > sms * (2 if d < 76 else 1)  # the bounds are taken
        o.sweep(1, 77, mask=O.MASK_SPLITMERGE)
        g.sweep(1, 77)
        assert dict(o.counters()) == dict(g.counters()), t
        zo, zbo = o.labels()
        zg, zbg = g.labels()
        assert o.K == g.K and np.array_equal(zo, zg) and np.array_equal(zbo, zbg), t
        merges += g.counters()["merges"]
    assert 0 < merges < K - 1
    g.close()
