"""What a context holds on the device, and what it leaves: creating one takes the tables that its sweeps need
and nothing for calls that may never be made; data of BF16X3 chains leave room for the input copies
of update_data and stage_data where the optional buffers would take it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _free():
    import torch

    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_a_context_holds_its_tables():
    import torch

    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    d, K = 144, 1000
    P.DPMM(P.PRIOR_NIW, 3, 4, 1.0).close()  # the library's own device image
    before = _free()
    g = P.DPMM(P.PRIOR_NIW, d, K, 1.0)
    taken = before - _free()
    g.close()
    nb = (d + 4) // 4
    E = 8 * nb * (nb + 1)  # entries of a sub-cluster's statistics
    ranges = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    tables = 8 * 2 * K * E + 3 * K * d * d * (8 + 4) + 8 * 2 * (ranges + K) * E  # statistics, W, records
    small = 3 * K * d * (8 * 6 + 4 * 4) + 3 * 8 * K * K  # a dozen tables of vectors, three of pairs
    assert taken <= tables + small + (16 << 20)


def test_input_copies_still_fit():
    import torch

    import __graft_entry__

    __graft_entry__.build()
    import paper_2204_08988_gb300 as P

    N, d = 4_000_003, 128
    host = torch.randn(N, d, generator=torch.Generator().manual_seed(1))
    X, pinned = host.numpy(), host.pin_memory()  # page-locked input is read in place
    y = (np.arange(N) % 4).astype(np.int32)
    zb = np.zeros(N, np.uint8)

    def chain(fill, how):
        hold = torch.empty(fill, dtype=torch.uint8, device="cuda") if fill else None
        g = P.DPMM(P.PRIOR_NIW, d, 8, 1.0, prec=P.PREC_BF16X3)
        try:
            g.set_data(pinned)
            left = _free()
            g.set_state(4, y, zb)
            getattr(g, how)(X)
            g.sweep(1, 5)
            return left, g.labels()
        finally:
            g.close()
            del hold
            torch.cuda.empty_cache()

    left, want = chain(0, "update_data")
    optional = 12 * N + N // 8 * 512  # the screened label step's buffers
    for how in ("update_data", "stage_data"):  # with room for 1.1 copies of the input beside what is needed
        room, got = chain(left + optional - X.nbytes * 11 // 10, how)
        assert room > X.nbytes and np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
