"""Which search serves a call, and that every one gives the same results: the
split search itself on batches the filter would take (mixed widths, graph, few
table rows), and the autotuner's trials on such a batch."""
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


def filtered(amp, g):
    return bool(g.tap(amp.abi.TAP_FILTERED, (1,), np.int32)[0])


def make(amp, dim, M, nlist, n, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    cent = r.standard_normal((nlist, dim)).astype(np.float32)
    books = (0.3 * r.standard_normal((M, 256, dim // M))).astype(np.float32)
    lo = r.integers(0, nlist, n).astype(np.int32)
    codes = r.integers(0, 256, (n, M)).astype(np.uint8)
    g = amp.Index(cent, books, codes, lo, device=0)
    return r, g, ivfpq.Index(cent, books, codes, lo)


def queries(r, o, nq):
    c = o.centroids
    return (c[r.integers(0, len(c), nq)] + 0.5 * r.standard_normal((nq, c.shape[1]))).astype(np.float32)


def same(got, want, what=""):
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a.cpu().numpy() if torch.is_tensor(a) else a, b, err_msg=what)


def test_split_search_by_itself(amp):
    """'split_scan' runs the two passes, wide pairs into a partial top-k and then the
    1..8-bit pairs, with the filtered search's results."""
    r, g, o = make(amp, 64, 16, 40, 30_000, 1)
    nq, nprobe = 1200, 20
    Q = queries(r, o, nq)
    widths = np.array([0, 4, 6, 8, 12, 16], np.uint8)[r.integers(0, 6, (nq, nprobe))]
    try:
        for k in (10, 40):
            for pol, bits in ((amp.policy("plain"), 0), (amp.policy("fixed", bits=8), 8),
                              (amp.policy("explicit", pair_bits=cuda(widths)), widths)):
                b = bits if np.isscalar(bits) else bits[:16]
                ri, rd = ivfpq.search(o, Q[:16], nprobe, k, bits=b)
                res = []
                for kern, f in (("filtered", True), ("split_scan", False), ("basic", False)):
                    g.set_kernel(kern)
                    res.append(g.search(cuda(Q), nprobe, k, pol))
                    assert filtered(amp, g) == f, (kern, k)
                    same([t[:16] for t in res[-1]], (ri, rd), kern)
                for i, d in res[1:]:
                    assert torch.equal(i, res[0][0]) and torch.equal(d, res[0][1])
    finally:
        g.close()


def test_graph_of_the_split_search_by_itself(amp):
    """Captured once, replayed with new queries and widths per pair."""
    r, g, o = make(amp, 32, 8, 64, 6000, 2)
    nq, nprobe, k = 40, 9, 40
    w = np.array([0, 4, 6, 8, 12, 16], np.uint8)
    qbuf, bbuf = cuda(queries(r, o, nq)), cuda(w[r.integers(0, 6, nq * nprobe)])
    g.set_kernel("split_scan")
    graph, ids, dists = g.capture_graph(qbuf, nprobe, k, amp.policy("explicit", pair_bits=bbuf))
    g.set_kernel("auto")
    try:
        for rep in range(3):
            Q2, b2 = queries(r, o, nq), w[r.integers(0, 6, nq * nprobe)]
            qbuf.copy_(cuda(Q2))
            bbuf.copy_(cuda(b2))
            ids.fill_(-7)
            graph.launch()
            torch.cuda.synchronize()
            same((ids, dists), ivfpq.search(o, Q2, nprobe, k, bits=b2.reshape(nq, nprobe)))
    finally:
        graph.close()
        g.close()


@pytest.mark.parametrize("M", [4, 8])
def test_narrow_pass_with_few_table_rows(amp, M):
    """Fewer table rows than warps, one row a warp, under 32- and 128-entry lists."""
    r, g, o = make(amp, 32, M, 16, 3000, M)
    Q = queries(r, o, 12)
    g.set_kernel("split_scan")
    try:
        for bits in (0, 4, 8):
            for k in (10, 100):
                pol = amp.policy("fixed", bits=bits) if bits else amp.policy("plain")
                same(g.search(cuda(Q), 6, k, pol), ivfpq.search(o, Q, 6, k, bits=bits), f"{bits} {k}")
                assert not filtered(amp, g)
    finally:
        g.close()


def test_filtered_whatever_the_batch(amp):
    """One query through the filter, with every width; fixed 4-bit tables, which it cannot serve, are scanned."""
    r, g, o = make(amp, 48, 12, 30, 4000, 5)
    Q = queries(r, o, 3)
    g.set_kernel("filtered")
    try:
        for nq in (1, 3):
            for bits in (0, 4, 6, 8, 12, 16):
                pol = amp.policy("fixed", bits=bits) if bits else amp.policy("plain")
                same(g.search(cuda(Q[:nq]), 7, 12, pol), ivfpq.search(o, Q[:nq], 7, 12, bits=bits), f"{nq} {bits}")
                assert filtered(amp, g) == (bits != 4)
    finally:
        g.close()


def test_autotuner_tries_each_search_once(amp):
    """On a batch the filter serves, the split search is tried by itself and the
    filtered search only as the automatic choice; what is installed is what ran."""
    r, g, o = make(amp, 64, 16, 40, 60_000, 3)
    Q = cuda(queries(r, o, 3000))
    A = amp.abi
    try:
        pol = amp.policy("plain")
        res = g.autotune(Q, 20, 10, pol, reps=1)
        tried = [(t[0], t[1]) for t in res]
        assert (A.KERNEL_AUTO, A.SCHED_AUTO) in tried and (A.KERNEL_SPLIT_SCAN, A.SCHED_LPT) in tried
        assert not any(t[0] == A.KERNEL_SPLIT for t in tried)
        assert len(set((t[0], t[1], t[3]) for t in res)) == len(res)
        best = min(res, key=lambda t: t[2])
        got = g.search(Q, 20, 10, pol)
        assert filtered(amp, g) == (best[0] == A.KERNEL_AUTO)
        same([t[:8] for t in got], ivfpq.search(o, Q[:8].cpu().numpy(), 20, 10, bits=0))
        with pytest.raises(amp.AnnsError):
            A.anns_set_option(g.handle, A.OPT_KERNEL, 7)
    finally:
        g.close()
