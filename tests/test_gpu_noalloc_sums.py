"""The allocation-free statistics: sums over many tiles keep 53 bits.  Every partial sum of these data is a
whole number below 2^53, and every tile's FP32 sums are exact, so the result is exact: one large
value in each tile (2^36) and odd and even small ones, whose sum leaves the 24 bits that lie below
the large ones' FP32 sum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,K,N", [(1, 1, 8_000_000), (2, 3, 3_000_011), (3, 1, 8_000_000)])
def test_whole_sums_are_exact(d, K, N):
    import torch

    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    g = torch.Generator(device="cuda").manual_seed(d)
    X = torch.randint(20_001, 32_767, (N, d), generator=g, device="cuda")
    X[::128] = 1 << 36
    z = torch.randint(0, K, (N,), generator=g, device="cuda", dtype=torch.int32)
    zb = torch.randint(0, 2, (N,), generator=g, device="cuda", dtype=torch.uint8) if K > 1 else torch.zeros(
        N, dtype=torch.uint8, device="cuda")
    out = [torch.full((2 * K * m,), -1.0, dtype=torch.float64, device="cuda") for m in (1, d, d * d)]
    P.dpmm_suffstats_noalloc(X.float(), z, zb, K, *out)
    slot = 2 * z.long() + zb.long()
    want = torch.stack([X[slot == s].sum(0) for s in range(2 * K)])
    assert int(want.max()) < 1 << 53
    assert torch.equal(out[0].long(), torch.bincount(slot, minlength=2 * K))
    assert torch.equal(out[1].view(2 * K, d).long(), want)
