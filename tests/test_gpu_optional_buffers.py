"""Label steps on a nearly full device: the buffers that only make them faster (the BF16X3
screening's, and the room for more undrawn clusters of the TF32 step's carry) are left out, the
data are accepted as before and the labels are the same whole numbers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,N,d,K", [("TF32", 300_001, 32, 60), ("BF16X3", 70_001, 100, 9)])
def test_labels_without_the_optional_buffers(prec, N, d, K):
    import torch

    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(d)
    mu = 0.4 * rng.standard_normal((K, d))
    X = (mu[rng.integers(0, K, N)] + rng.standard_normal((N, d))).astype(np.float32)

    def labels():
        g = P.DPMM(P.PRIOR_NIW, d, 64, 1.0, prec=getattr(P, "PREC_" + prec), psi0=np.eye(d))
        try:
            g.set_data(X)
            g.set_state(K, (np.arange(N) % K).astype(np.int32), np.zeros(N, np.uint8))
            g.sweep(3, 7)
            return g.labels()
        finally:
            g.close()

    want = labels()
    free, _ = torch.cuda.mem_get_info()
    fill = torch.empty(free - (1000 << 20), dtype=torch.uint8, device="cuda")  # less than a GiB is left
    got = labels()
    del fill
    torch.cuda.empty_cache()
    assert np.array_equal(want[0], got[0]) and np.array_equal(want[1], got[1])
