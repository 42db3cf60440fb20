"""Dense multinomial data of up to 256 categories are taken with fractional values (weighted counts):
the split and merge ratios use the sums as they are.  Two halves of one cluster, beta not uniform:
the merge's log ratio is far above 0, and far below it with the categories' fractions dropped."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,N", [(40, 600), (256, 901)])
def test_fractional_counts_merge(d, N):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(d)
    beta = rng.uniform(0.5, 1.5, d)
    X = rng.gamma(0.3, size=(N, d)).astype(np.float32)
    z = (np.arange(N) % 2).astype(np.int32)
    zb = (np.arange(N) // 2 % 2).astype(np.uint8)
    lgam = np.vectorize(math.lgamma)

    def marginal(c, total):
        return math.lgamma(beta.sum()) - math.lgamma(beta.sum() + total) + (lgam(beta + c) - lgam(beta)).sum()

    def ratio(whole):
        c = [X[z == k].astype(np.float64).sum(0) for k in (0, 1)]
        c.append(c[0] + c[1])
        m = [marginal(v, (np.floor(v) if whole else v).sum()) for v in c]
        n0, n1, a = (z == 0).sum(), (z == 1).sum(), 1.0
        return (-math.log(a) + math.lgamma(N) - math.lgamma(n0) - math.lgamma(n1) + m[2] - m[0] - m[1] + math.lgamma(a)
                - math.lgamma(a + N) + math.lgamma(a / 2 + n0) + math.lgamma(a / 2 + n1) - 2 * math.lgamma(a / 2))

    assert ratio(False) > 1.0 and ratio(True) < -60.0  # -36.8 <= log u < 0
    g = P.DPMM(P.PRIOR_DIRICHLET, d, 8, 1.0, prec=P.PREC_FP32, beta=beta)
    g.set_data(X)
    g.set_state(2, z, zb)
    g.set_mask(4)
    g.sweep(1, 3)
    assert g.counters()["merges"] == 1 and g.K == 1
    g.close()
