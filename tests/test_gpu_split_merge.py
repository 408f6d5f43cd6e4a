"""The merge of several blocks' partial results of one query (small batches):
ranks by binary search in the sorted parts, with equal distances across and
within parts, fewer vectors than k, per-query k and nprobe, up to 32 parts of 32."""
import numpy as np
import pytest

from oracle import ivfpq

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,nprobe,k", [(1, 32, 32), (2, 40, 32), (13, 31, 32), (19, 33, 32), (7, 3, 5), (300, 2, 31)])
@pytest.mark.parametrize("ties", [False, True])
def test_parts_are_merged_by_distance_and_id(nq, nprobe, k, ties):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_07156_gb300 as amp
    r = np.random.Generator(np.random.PCG64(nq * 7 + k))
    nlist, dim, M = 48, 32, 8
    cent = r.standard_normal((nlist, dim)).astype(np.float32)
    books = (0.3 * r.standard_normal((M, 256, dim // M))).astype(np.float32)
    lo = np.repeat(np.arange(nlist, dtype=np.int32), r.integers(0, 40, nlist))
    codes = r.integers(0, 256, (len(lo), M)).astype(np.uint8)
    if ties:  # three distinct centroids, two distinct codes: almost every distance is shared
        cent = cent[np.arange(nlist) % 3].copy()
        codes = codes[np.arange(len(lo)) % 2].copy()
    ids = r.permutation(len(lo)).astype(np.int64)
    Q = (cent[r.integers(0, nlist, nq)] + 0.4 * r.standard_normal((nq, dim))).astype(np.float32)
    npq = r.integers(0, nprobe + 1, nq).astype(np.int32)
    kpq = r.integers(0, k + 1, nq).astype(np.int32)
    g = amp.Index(cent, books, codes, lo, ids=ids, device=0)
    o = ivfpq.Index(cent, books, codes, lo, ids)
    cuda = lambda a: torch.from_numpy(a).to("cuda:0")  # noqa: E731
    try:
        for pol, b in ((amp.policy("plain"), 0), (amp.policy("fixed", bits=16), 16)):
            for kw in ({}, dict(nprobe_per_q=npq, k_per_q=kpq)):
                i, d = g.search(cuda(Q), nprobe, k, pol, **{f: cuda(v) for f, v in kw.items()})
                ri, rd = ivfpq.search(o, Q, nprobe, k, bits=b, **kw)
                np.testing.assert_array_equal(i.cpu().numpy(), ri)
                np.testing.assert_array_equal(d.cpu().numpy(), rd)
    finally:
        g.close()
