"""The allocation-free statistics kernel over the sizes where it can go wrong: every width of
its instantiations and their edges, one slot and all of them, tiles and slices that are
empty, ragged or all one slot's, and sums that leave FP32's range (added up in FP64 then).

Bound: a tile's points of one slot are FP32 sums of at most 128 products (each partial sum
rounded once: 128 x 2^-24 of the sum of the magnitudes), added up to at least 46 bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 128 * 2.0 ** -24


def _check(X, K, z, zb):
    import torch

    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    d = X.shape[1]
    out = [torch.full((2 * K * m,), -1.0, dtype=torch.float64, device="cuda") for m in (1, d, d * d)]
    P.dpmm_suffstats_noalloc(torch.from_numpy(X).cuda(), torch.from_numpy(z).cuda(), torch.from_numpy(zb).cuda(), K, *out)
    torch.cuda.synchronize()
    n, sx, sxx = (o.cpu().numpy() for o in out)
    sx, sxx = sx.reshape(2 * K, d), sxx.reshape(2 * K, d, d)
    Y = X.astype(np.float64)
    for s in range(2 * K):
        A = Y[(z == s // 2) & (zb == s % 2)]
        assert n[s] == len(A)
        M = np.abs(A)
        assert np.all(np.abs(sx[s] - A.sum(0)) <= EPS * M.sum(0))
        assert np.all(np.abs(sxx[s] - A.T @ A) <= EPS * (M.T @ M))


@pytest.mark.parametrize("d,K,N", [(1, 1, 1), (2, 16, 127), (3, 2, 129), (4, 1, 40_001), (5, 3, 4_097), (8, 16, 50_000),
                                   (9, 7, 20_003), (16, 2, 33_333), (17, 5, 12_345), (31, 16, 70_001), (32, 1, 9_999),
                                   (32, 16, 200_003)])
def test_sizes(d, K, N):
    rng = np.random.default_rng(d * 100 + K)
    X = (rng.standard_normal((N, d)) * 3 + 1).astype(np.float32)
    z = rng.integers(0, K + 1, N).astype(np.int32) if K > 1 else np.zeros(N, np.int32)  # K: ignored
    zb = rng.integers(0, 2, N).astype(np.uint8)
    if N > 10_000:  # a stretch of whole tiles of one slot, and one without any of it
        z[2_000:6_000] = 0
        zb[2_000:4_500] = 1
        z[6_000:9_000] = K - 1
    _check(X, K, z, zb)


def test_sums_beyond_fp32_are_finite():
    rng = np.random.default_rng(1)
    X = (rng.standard_normal((30_000, 6)) * 1e18).astype(np.float32)  # products near 1e36, sums near 1e40
    _check(X, 1, np.zeros(len(X), np.int32), np.zeros(len(X), np.uint8))


def test_an_infinity_stays_in_its_own_entries():
    import torch

    import paper_2204_08988_gb300 as P

    d, N = 5, 3_000
    X = np.ones((N, d), np.float32)
    X[1234, 2] = np.inf
    out = [torch.zeros(m, dtype=torch.float64, device="cuda") for m in (4, 4 * d, 4 * d * d)]
    z = (np.arange(N) % 2).astype(np.int32)
    P.dpmm_suffstats_noalloc(torch.from_numpy(X).cuda(), torch.from_numpy(z).cuda(),
                             torch.zeros(N, dtype=torch.uint8, device="cuda"), 2, *out)
    torch.cuda.synchronize()
    sxx = out[2].cpu().numpy().reshape(4, d, d)
    want = np.full((d, d), 1500.0)
    want[2, :] = want[:, 2] = np.inf
    assert np.array_equal(sxx[0], want) and np.array_equal(sxx[2], np.full((d, d), 1500.0))
