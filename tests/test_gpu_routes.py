"""The automatic choice of a search: whatever it picks, results are the oracle's,
on an index the filter cannot serve (a codebook entry that no vector uses is not
finite) and on one it can; the counts of an uneven batch are taken into account
where they are on the host."""
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


def make(amp, rows, n=24_000, nlist=80, dim=48, M=12):
    r = np.random.Generator(np.random.PCG64(n + rows))
    cent = r.standard_normal((nlist, dim)).astype(np.float32)
    books = (0.3 * r.standard_normal((M, 256, dim // M))).astype(np.float32)
    lo = (r.random(n) ** 2 * nlist).astype(np.int32)          # uneven lists
    codes = r.integers(0, 255, (n, M)).astype(np.uint8)
    b = books.copy()
    if not rows:
        b[0, 255, 1] = np.inf             # no vector has code 255
    g = amp.Index(cent, b, codes, lo, device=0)
    return r, g, ivfpq.Index(cent, books, codes, lo)


@pytest.mark.parametrize("rows", [False, True])
@pytest.mark.parametrize("nq", [1, 16, 130])
@pytest.mark.parametrize("k", [10, 100])
def test_every_route_gives_the_oracles_results(amp, rows, nq, k):
    r, g, o = make(amp, rows)
    Q = (o.centroids[r.integers(0, 80, nq)] + 0.5 * r.standard_normal((nq, 48))).astype(np.float32)
    try:
        for nprobe in (3, 40):
            npq = r.integers(0, nprobe + 1, nq).astype(np.int32)
            widths = np.array([0, 4, 6, 8, 12, 16], np.uint8)[r.integers(0, 6, (nq, nprobe))]
            for pol, bits in ((amp.policy("plain"), 0), (amp.policy("fixed", bits=4), 4), (amp.policy("fixed", bits=8), 8),
                              (amp.policy("fixed", bits=12), 12),
                              (amp.policy("explicit", pair_bits=cuda(widths)), widths)):
                if not rows and not (np.isscalar(bits) and bits == 0):
                    continue          # tables of that codebook are not finite
                ri, rd = ivfpq.search(o, Q, nprobe, k, bits=bits)
                ui, ud = ivfpq.search(o, Q, nprobe, k, bits=bits, nprobe_per_q=npq)
                for sched in ("auto", "lpt"):
                    g.set_schedule(sched)
                    i, d = g.search(cuda(Q), nprobe, k, pol)
                    if not rows:
                        assert g.tap(amp.abi.TAP_FILTERED, (1,), np.int32)[0] == 0
                    np.testing.assert_array_equal(i.cpu().numpy(), ri)
                    np.testing.assert_array_equal(d.cpu().numpy(), rd)
                    i, d = g.search(cuda(Q), nprobe, k, pol, nprobe_per_q=cuda(npq))
                    np.testing.assert_array_equal(i.cpu().numpy(), ui)
                    np.testing.assert_array_equal(d.cpu().numpy(), ud)
                    i, d = g.search_host(Q, nprobe, k, pol, nprobe_per_q=npq)
                    np.testing.assert_array_equal(i, ui)
                    np.testing.assert_array_equal(d, ud)
    finally:
        g.close()


def test_counts_on_the_host_decide(amp):
    """The same batch with every count at nprobe, or at 1: filtered or not, as its real size pays."""
    r, g, o = make(amp, True, n=120_000, nlist=100)
    nq, nprobe = 2000, 64
    Q = (o.centroids[r.integers(0, 100, nq)] + 0.5 * r.standard_normal((nq, 48))).astype(np.float32)
    try:
        got = {}
        for count in (nprobe, 1):
            npq = np.full(nq, count, np.int32)
            i, d = g.search_host(Q, nprobe, 10, amp.policy("plain"), nprobe_per_q=npq)
            got[count] = int(g.tap(amp.abi.TAP_FILTERED, (1,), np.int32)[0])
            ri, rd = ivfpq.search(o, Q[:10], nprobe, 10, bits=0, nprobe_per_q=npq[:10])
            np.testing.assert_array_equal(i[:10], ri)
            np.testing.assert_array_equal(d[:10], rd)
        assert got == {nprobe: 1, 1: 0}
    finally:
        g.close()
