"""The filter's device memory: a workspace limit and a failed allocation make
that one call scan, a limit of 0 gives the decoded rows back, a captured graph
keeps the rows it was captured with, and results are the same throughout."""
import gc

import numpy as np
import pytest

from oracle import ivfpq

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amp():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_07156_gb300 as m
    return m


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def make(amp, dim, M, nlist, n, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    cent = r.standard_normal((nlist, dim)).astype(np.float32)
    books = (0.3 * r.standard_normal((M, 256, dim // M))).astype(np.float32)
    lo = r.integers(0, nlist, n).astype(np.int32)
    codes = r.integers(0, 256, (n, M)).astype(np.uint8)
    g = amp.Index(cent, books, codes, lo, device=0)
    return r, g, ivfpq.Index(cent, books, codes, lo)


def filtered(amp, g):
    return bool(g.tap(amp.abi.TAP_FILTERED, (1,), np.int32)[0])


def used():
    torch.cuda.synchronize()
    gc.collect()
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_limit_and_rows_given_back(amp):
    r, g, o = make(amp, 64, 16, 64, 400_000, 1)
    nq, nprobe, k = 2000, 20, 10
    Q = cuda((o.centroids[r.integers(0, 64, nq)] + 0.5 * r.standard_normal((nq, 64))).astype(np.float32))
    want = ivfpq.search(o, Q[:8].cpu().numpy(), nprobe, k, bits=0)
    g.set_kernel("filtered")

    def check(f):
        i, d = g.search(Q, nprobe, k, amp.policy("plain"))
        assert filtered(amp, g) == f
        np.testing.assert_array_equal(i[:8].cpu().numpy(), want[0])
        np.testing.assert_array_equal(d[:8].cpu().numpy(), want[1])
        return i, d
    try:
        first = check(True)
        g.set_filter_bytes(1000)                    # no workspace fits: scanned
        second = check(False)
        assert torch.equal(first[0], second[0]) and torch.equal(first[1], second[1])
        g.set_filter_bytes(1 << 35)
        check(True)
        graph, ids, dists = g.capture_graph(Q, nprobe, k, amp.policy("plain"))
        before = used()
        g.set_filter_bytes(0)                       # the graph keeps the rows
        check(False)
        ids.fill_(-7)
        dists.fill_(-7)
        graph.launch()
        torch.cuda.synchronize()
        assert torch.equal(ids, first[0]) and torch.equal(dists, first[1])
        graph.close()
        assert used() <= before - 400_000 * 64 * 2  # given back with the graph
        check(False)
        g.set_filter_bytes(1 << 35)                 # formed again
        check(True)
        with pytest.raises(amp.AnnsError):
            g.set_filter_bytes(-1)
    finally:
        g.close()


def test_allocation_that_fails(amp):
    """A workspace larger than the device (about 330 GB of slot rows, with the limit raised): the
    allocation fails, the call scans with the oracle's results, smaller calls are filtered before and
    after, and a captured graph of the large batch scans."""
    r, g, o = make(amp, 4096, 16, 128, 2000, 2)
    nq, nprobe, k = 160_000, 128, 1
    Q = torch.randn(nq, 4096, device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(3))
    g.set_kernel("filtered")
    g.set_filter_bytes(1 << 50)
    want = ivfpq.search(o, Q[:4].cpu().numpy(), nprobe, k, bits=0)

    def small():
        i, d = g.search(Q[:300], nprobe, k, amp.policy("plain"))
        assert filtered(amp, g)
        np.testing.assert_array_equal(i[:4].cpu().numpy(), want[0])
    try:
        small()
        for _ in range(2):
            i, d = g.search(Q, nprobe, k, amp.policy("plain"))
            assert not filtered(amp, g)
            np.testing.assert_array_equal(i[:4].cpu().numpy(), want[0])
            np.testing.assert_array_equal(d[:4].cpu().numpy(), want[1])
            small()
        graph, ids, dists = g.capture_graph(Q, nprobe, k, amp.policy("plain"))
        ids.fill_(-7)
        graph.launch()
        torch.cuda.synchronize()
        assert torch.equal(ids, i) and torch.equal(dists, d)
        graph.close()
    finally:
        g.close()
