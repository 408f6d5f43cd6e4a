"""The filtered search of mixed table widths with k <= 32, the learned policy's
way on large batches: queries with FP32 survivors only settled by a warp, the
others by a block, 4-bit pairs (of every rank, the nearest among them) marked and
scanned eight to a word under the filter's bound, and queries with more
candidates than fit handed to the scan. Every call asserts that it was filtered
and equals the oracle on a sample and the query-major search on the whole batch."""
import numpy as np
import pytest

from oracle import ivfpq

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NLIST, DIM, M = 64, 64, 16


@pytest.fixture(scope="module")
def amp():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_07156_gb300 as m
    return m


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


@pytest.fixture(scope="module")
def pair(amp):
    r = np.random.Generator(np.random.PCG64(17))
    cent = r.standard_normal((NLIST, DIM)).astype(np.float32)
    books = (0.3 * r.standard_normal((M, 256, DIM // M))).astype(np.float32)
    lo = r.integers(0, NLIST, 160_000).astype(np.int32)
    codes = r.integers(0, 256, (len(lo), M)).astype(np.uint8)
    for l in (3, 11):                     # 6000 equal vectors each: more candidates than fit
        i = np.flatnonzero(lo == l)
        extra = np.flatnonzero(lo == l + 20)[:6000 - len(i)]
        lo[extra] = l
        codes[lo == l] = codes[i[0]]
    g = amp.Index(cent, books, codes, lo, device=0)
    yield r, g, ivfpq.Index(cent, books, codes, lo)
    g.close()


def run(amp, g, o, Q, nprobe, k, pol, bits, **kw):
    kwd = {f: cuda(v) for f, v in kw.items()}
    g.set_kernel("filtered")
    try:
        i, d = g.search(cuda(Q), nprobe, k, pol, **kwd)
        assert g.tap(amp.abi.TAP_FILTERED, (1,), np.int32)[0] == 1
        amp.abi.anns_sync_status(g.handle)
        if bits is None:
            bits = g.tap(amp.abi.TAP_BITS, (len(Q), nprobe), np.uint8)
        g.set_kernel("basic")
        bi, bd = g.search(cuda(Q), nprobe, k, pol, **kwd)
        assert torch.equal(i, bi) and torch.equal(d, bd)
        s = slice(0, 10)
        ri, rd = ivfpq.search(o, Q[s], nprobe, k, bits=bits[s], **{f: v[s] for f, v in kw.items()})
        np.testing.assert_array_equal(i[s].cpu().numpy(), ri)
        np.testing.assert_array_equal(d[s].cpu().numpy(), rd)
    finally:
        g.set_kernel("auto")


@pytest.mark.parametrize("k", [1, 10, 32])
@pytest.mark.parametrize("uneven", [False, True])
def test_explicit_widths(amp, pair, k, uneven):
    r, g, o = pair
    nq, nprobe = 4000, 40
    Q = (o.centroids[r.integers(0, NLIST, nq)] + 0.5 * r.standard_normal((nq, DIM))).astype(np.float32)
    Q[:4] = o.centroids[[3, 11, 3, 11]]
    bits = r.choice(np.array([0, 4, 4, 6, 8, 12, 16], np.uint8), size=(nq, nprobe))
    bits[4:nq // 2, 0] = 4                # the nearest pair on a 4-bit table
    bits[nq // 2:] = np.where(bits[nq // 2:] > 4, 0, bits[nq // 2:])   # FP32 and 4-bit pairs only
    kw = {}
    if uneven:
        kw = dict(nprobe_per_q=r.integers(0, nprobe + 1, nq).astype(np.int32),
                  k_per_q=r.integers(0, k + 1, nq).astype(np.int32))
        kw["nprobe_per_q"][:4] = nprobe
    run(amp, g, o, Q, nprobe, k, amp.policy("explicit", pair_bits=cuda(bits)), bits, **kw)


@pytest.mark.parametrize("k", [10, 32])
@pytest.mark.parametrize("width_map", [False, True])
def test_learned_widths(amp, pair, k, width_map):
    r, g, o = pair
    nq, nprobe = 4000, 40
    p = {f: r.uniform(-1, 1, s).astype(np.float32) for f, s in amp._PRED_SHAPES.items()}
    p["inv_std"] = np.abs(p["inv_std"]) + 0.1
    g.set_predictor(p)
    Q = (o.centroids[r.integers(0, NLIST, nq)] + 0.5 * r.standard_normal((nq, DIM))).astype(np.float32)
    run(amp, g, o, Q, nprobe, k, amp.policy("mlp", margin=0.1, width_map=width_map), None)
