"""Failure detection of the filter's GEMM without a fault: with a wait limit of
one clock cycle its main-loop waits run out. Fewer than 256 lists keep the FP32
coarse stage on the CUDA cores, so no other kernel of the search has such waits.
The timeout is reported once, the copies in flight are waited for (D = 96: two
chunks, all issued before another role gives up; D = 960: the ring has wrapped),
and with the default limit back the index gives the oracle's results."""
import numpy as np
import pytest

from oracle import ivfpq

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,M", [(96, 48), (960, 120)])
def test_filter_wait_timeout_is_reported_and_recovers(dim, M):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_07156_gb300 as amp
    from paper_2606_07156_gb300 import abi
    r = np.random.Generator(np.random.PCG64(dim))
    nlist, n, nq, nprobe, k = 60, 90_000, 1500, 24, 10
    cent = r.standard_normal((nlist, dim)).astype(np.float32)
    books = (0.3 * r.standard_normal((M, 256, dim // M))).astype(np.float32)
    lo = r.integers(0, nlist, n).astype(np.int32)
    codes = r.integers(0, 256, (n, M)).astype(np.uint8)
    Q = (cent[r.integers(0, nlist, nq)] + 0.5 * r.standard_normal((nq, dim))).astype(np.float32)
    g = amp.Index(cent, books, codes, lo, device=0)
    o = ivfpq.Index(cent, books, codes, lo)
    Qd = torch.from_numpy(Q).to("cuda:0")
    ri, rd = ivfpq.search(o, Q[:8], nprobe, k, bits=0)
    try:
        g.search(Qd, nprobe, k, amp.policy("plain"))
        abi.anns_sync_status(g.handle)                      # no timeout with the default limit
        abi.anns_set_option(g.handle, abi.OPT_WAIT_CYCLES, 1)
        for _ in range(2):
            g.search(Qd, nprobe, k, amp.policy("plain"))
            with pytest.raises(amp.AnnsError) as e:
                abi.anns_sync_status(g.handle)
            assert e.value.code == -4 and "ran out" in str(e.value)
            abi.anns_sync_status(g.handle)                  # read and cleared
        abi.anns_set_option(g.handle, abi.OPT_WAIT_CYCLES, 0)
        ids, dists = g.search(Qd, nprobe, k, amp.policy("plain"))
        abi.anns_sync_status(g.handle)
        np.testing.assert_array_equal(ids.cpu().numpy()[:8], ri)
        np.testing.assert_array_equal(dists.cpu().numpy()[:8], rd)
        g.set_kernel("basic")
        bi, bd = g.search(Qd, nprobe, k, amp.policy("plain"))
        assert torch.equal(ids, bi) and torch.equal(dists, bd)
    finally:
        g.close()
