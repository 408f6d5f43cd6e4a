"""The tensor-core filter in front of the exact rules: searches it serves equal
the CPU oracle's bit for bit, at the edges of its tiles (256 vectors, 128
queries a group, 16-column steps, 64-element K chunks), for every table width,
and for queries it hands to the scanning kernel (more candidates than fit, NaN).
"""
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


def make_index(amp, dim, M, sizes, seed, spread=0.35):
    """Random index with the given list sizes; codes are the entries nearest to random residuals' signs."""
    r = np.random.Generator(np.random.PCG64(seed))
    nlist = len(sizes)
    cent = r.standard_normal((nlist, dim)).astype(np.float32)
    books = (spread * r.standard_normal((M, 256, dim // M))).astype(np.float32)
    lo = np.repeat(np.arange(nlist, dtype=np.int32), sizes)
    r.shuffle(lo)
    codes = r.integers(0, 256, (len(lo), M)).astype(np.uint8)
    ids = r.permutation(10 * len(lo))[:len(lo)].astype(np.int64)
    g = amp.Index(cent, books, codes, lo, ids=ids, device=0)
    g.set_kernel("split")  # filtered at these sizes whatever the tables (automatic: small quantised batches are grouped)
    return r, g, ivfpq.Index(cent, books, codes, lo, ids)


def queries(r, o, nq, noise=0.5):
    c = o.centroids
    return (c[r.integers(0, len(c), nq)] + noise * r.standard_normal((nq, c.shape[1]))).astype(np.float32)


def check(amp, g, o, Q, nprobe, k, pol, bits, **kw):
    ids, dists = g.search(cuda(Q), nprobe, k, pol, **{f: cuda(v) for f, v in kw.items()})
    torch.cuda.synchronize()
    amp.abi.anns_sync_status(g.handle)
    ri, rd = ivfpq.search(o, Q, nprobe, k, bits=bits, **kw)
    np.testing.assert_array_equal(ids.cpu().numpy(), ri)
    np.testing.assert_array_equal(dists.cpu().numpy(), rd)


SIZES = [0, 1, 31, 64, 65, 127, 128, 129, 255, 256, 257, 300, 511, 513, 900, 3000, 20000]


@pytest.mark.parametrize("dim,M", [(16, 8), (64, 16), (96, 48), (100, 20), (136, 17), (256, 32), (960, 120)])
@pytest.mark.parametrize("bits", [0, 8, 12])
def test_tile_edges(amp, dim, M, bits):
    r, g, o = make_index(amp, dim, M, SIZES, dim + M)
    pol = amp.policy("fixed", bits=bits) if bits else amp.policy("plain")
    try:
        for nq, nprobe, k in ((1, 16, 10), (17, 9, 1), (145, 16, 33)):
            check(amp, g, o, queries(r, o, nq), nprobe, k, pol, bits)
    finally:
        g.close()


@pytest.mark.parametrize("k", [10, 100, 128])
@pytest.mark.parametrize("kern", ["auto", "split"])
def test_uneven_batches_and_widths(amp, k, kern):
    """Per-query nprobe and k (0 included) with a table width per pair, 4-bit pairs of every rank among them."""
    r, g, o = make_index(amp, 64, 16, [400 + 37 * i for i in range(24)], 5)
    nq, nprobe = 150, 20
    Q = queries(r, o, nq)
    npq = r.integers(0, nprobe + 1, nq).astype(np.int32)
    kpq = r.integers(0, k + 1, nq).astype(np.int32)
    bits = r.choice(np.array([0, 4, 4, 6, 8, 12, 16], np.uint8), size=(nq, nprobe))
    g.set_kernel(kern)
    try:
        check(amp, g, o, Q, nprobe, k, amp.policy("explicit", pair_bits=cuda(bits)), bits, nprobe_per_q=npq, k_per_q=kpq)
        for cl in ("fp16", "bf16"):
            check(amp, g, o, Q, nprobe, k, amp.policy("plain", cl=cl), 0, nprobe_per_q=npq, k_per_q=kpq)
            check(amp, g, o, Q, nprobe, k, amp.policy("fixed", bits=6, cl=cl), 6)
    finally:
        g.close()


def test_queries_left_to_the_scan(amp):
    """Lists of equal vectors (every one a candidate), a NaN query and huge values: scanned, same results."""
    r = np.random.Generator(np.random.PCG64(3))
    cent = r.standard_normal((6, 32)).astype(np.float32)
    books = (0.3 * r.standard_normal((8, 256, 4))).astype(np.float32)
    lo = np.repeat(np.arange(6, dtype=np.int32), [6000, 500, 5000, 300, 700, 900])
    codes = r.integers(0, 256, (len(lo), 8)).astype(np.uint8)
    codes[lo == 0] = 7
    codes[lo == 2] = 9
    g = amp.Index(cent, books, codes, lo, device=0)
    g.set_kernel("split")
    o = ivfpq.Index(cent, books, codes, lo)
    Q = (cent[r.integers(0, 6, 40)] + 0.1 * r.standard_normal((40, 32))).astype(np.float32)
    Q[3] = cent[0]
    Q[4] = cent[2]
    Q[7] *= np.float32(1e18)
    try:
        for bits in (0, 8, 16):
            check(amp, g, o, Q, 6, 10, amp.policy("fixed", bits=bits) if bits else amp.policy("plain"), bits)
        Q2 = Q.copy()
        Q2[5, 3] = np.nan
        ids, dists = g.search(cuda(Q2), 6, 10, amp.policy("plain"))
        ids, dists = ids.cpu().numpy(), dists.cpu().numpy()
        g.set_kernel("basic")
        want_i, want_d = (t.cpu().numpy() for t in g.search(cuda(Q2), 6, 10, amp.policy("plain")))
        np.testing.assert_array_equal(ids, want_i)
        np.testing.assert_array_equal(dists, want_d)
    finally:
        g.close()


def test_scales(amp):
    """Bounds hold for tiny and large magnitudes and for data far from the origin."""
    for scale, shift in ((1e-12, 0.0), (1e12, 0.0), (1.0, 300.0), (50.0, 128.0)):
        r = np.random.Generator(np.random.PCG64(11))
        cent = (scale * r.standard_normal((12, 48)) + shift).astype(np.float32)
        books = (0.3 * scale * r.standard_normal((12, 256, 4))).astype(np.float32)
        lo = r.integers(0, 12, 20000).astype(np.int32)
        codes = r.integers(0, 256, (20000, 12)).astype(np.uint8)
        g = amp.Index(cent, books, codes, lo, device=0)
        g.set_kernel("split")
        o = ivfpq.Index(cent, books, codes, lo)
        Q = (cent[r.integers(0, 12, 33)] + 0.4 * scale * r.standard_normal((33, 48))).astype(np.float32)
        try:
            check(amp, g, o, Q, 10, 10, amp.policy("plain"), 0)
            check(amp, g, o, Q, 10, 10, amp.policy("fixed", bits=8), 8)
        finally:
            g.close()
