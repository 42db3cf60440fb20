"""The getters: get_stats where the unpacked statistics leave the device in more than one piece (compressed rows of as
many clusters as the context holds), and with outputs left out: the sums are those of the labels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,K,K_max", [(300, 4, 4), (257, 1, 1), (1000, 7, 9)])
def test_compressed_rows(d, K, K_max):
    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(d)
    N = 500
    X = rng.poisson(0.05, (N, d)).astype(np.int32)
    z = (np.arange(N) % K).astype(np.int32)
    zb = rng.integers(0, 2, N).astype(np.uint8)
    g = P.DPMM(P.PRIOR_DIRICHLET, d, K_max, 1.0, prec=P.PREC_FP32, beta=np.ones(d))
    g.set_data(X)
    g.set_state(K, z, zb)
    n, sx, _ = g.stats()
    for k in range(K):
        for s, at in enumerate([z == k, (z == k) & (zb == 0), (z == k) & (zb == 1)]):
            assert n[3 * k + s] == at.sum() and np.array_equal(sx[3 * k + s], X[at].sum(0))
    g.close()


@pytest.mark.parametrize("d,K,K_max", [(1, 3, 3), (2, 1, 1), (33, 40, 1000)])
def test_gaussian(d, K, K_max):
    import ctypes as C

    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    rng = np.random.default_rng(d)
    N = 2_000
    X = rng.standard_normal((N, d)) + 5.0
    z = (np.arange(N) % K).astype(np.int32)
    zb = rng.integers(0, 2, N).astype(np.uint8)
    g = P.DPMM(P.PRIOR_NIW, d, K_max, 1.0, prec=P.PREC_FP64_PLAIN)
    g.set_data(X)
    g.set_state(K, z, zb)
    n, sx, sxx = g.stats()
    for k in range(K):
        for s, at in enumerate([z == k, (z == k) & (zb == 0), (z == k) & (zb == 1)]):
            assert n[3 * k + s] == at.sum()
            assert np.allclose(sx[3 * k + s], X[at].sum(0), rtol=1e-12, atol=1e-12)
            assert np.allclose(sxx[3 * k + s], X[at].T @ X[at], rtol=1e-12, atol=1e-12)
    only = np.zeros(3 * K_max * d)
    Kout = C.c_int()
    assert P.load().dpmm_get_stats(g.h, C.byref(Kout), None, only.ctypes.data_as(C.c_void_p), None, None) == 0
    assert Kout.value == K and np.array_equal(only[: 3 * K * d], sx.reshape(-1))
    g.close()


def test_more_contexts_than_slots():
    """Getters of 300 contexts alive at once, and of contexts created as others go, from several threads."""
    import concurrent.futures as cf

    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    def chain(i):
        g = P.DPMM(P.PRIOR_NIW, 2, 8, 1.0)
        n = 16 + i % 7
        g.set_data(np.random.default_rng(i).standard_normal((n, 2)))
        g.set_state(1 + i % 5, (np.arange(n) % (1 + i % 5)).astype(np.int32), np.zeros(n, np.uint8))
        g.set_iter(i)
        return g

    def seen(g):
        return g.info() + (g.stats()[0][0::3].sum(),)

    held = [chain(i) for i in range(300)]
    assert [seen(g) for g in held] == [(1 + i % 5, i, 16 + i % 7) for i in range(300)]
    for g in held[::3]:
        g.close()

    def work(i):
        g = chain(i)
        out = seen(g)
        g.close()
        return out

    with cf.ThreadPoolExecutor(8) as ex:
        assert list(ex.map(work, range(64))) == [(1 + i % 5, i, 16 + i % 7) for i in range(64)]
    assert [seen(g) for g in held[1::3]] == [(1 + i % 5, i, 16 + i % 7) for i in range(1, 300, 3)]
