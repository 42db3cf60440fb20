"""The FP64 factorisation of the parameter draws against the oracle: dimensions around the panels
of four pivots and the warps' 32 rows, and scales whose pivots' reciprocals leave the FP32 range.
Clusters are near-spherical with 20 points and more per dimension, so the factors' condition is
below 10 and d^2 roundings of 2^-53 keep every entry within 2e-11 of the largest."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,scale", [(1, 1.0), (3, 1.0), (4, 1.0), (5, 1.0), (8, 1.0), (9, 1.0), (31, 1.0), (32, 1.0), (33, 1.0),
                                     (66, 1.0), (129, 1.0), (6, 1e100), (6, 1e-100), (5, 1e152), (5, 1e-152)])
def test_draws_match_oracle(d, scale):
    rng = np.random.default_rng(d)
    K, N = 2, 60 * d + 40
    y = (np.arange(N) % K).astype(np.int32)
    zb = (rng.random(N) < 0.5).astype(np.uint8)
    X = (rng.standard_normal((N, d)) + 3.0 * rng.standard_normal((K, d))[y]) * scale
    prior = dict(kappa0=1.0, m0=np.zeros(d), nu0=d + 3.0, psi0=np.eye(d) * scale * scale)
    o = O.Oracle(O.NIW, d, 4, 2.0, **prior)
    o.set_data(X)
    o.set_state(K, y, zb)
    o.iter = 3
    o.draw_params(99)
    want = o.params()
    assert all(np.isfinite(want[k]).all() for k in ("logw", "mu", "W", "logdetW"))

    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    g = P.DPMM(P.PRIOR_NIW, d, 4, 2.0, prec=P.PREC_FP64_PLAIN, **prior)
    g.set_data(X)
    g.set_state(K, y, zb)
    g.set_iter(3)
    g.set_mask(1)
    g.sweep(1, 99)
    if scale == 1e152:  # the product of two first moments overflows ahead of the factorisation: refused, as ever
        with pytest.raises(P.DPMMError, match="ENUMERIC"):
            g.params()
        return
    got = g.params()
    g.close()
    for key in ("logw", "mu", "W", "logdetW"):
        assert np.abs(want[key] - got[key]).max() <= 1e-9 * np.abs(want[key]).max(), key
