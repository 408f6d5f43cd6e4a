"""Index build and export move the codes in pieces of 2^24 vectors: an index a
little larger than one piece exports what it was built from, from host and
device arrays, and a search finds vectors on both sides of the seam."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("device", [False, True])
def test_more_than_one_piece(device):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_07156_gb300 as amp
    r = np.random.Generator(np.random.PCG64(5))
    n, nlist, dim, M = (1 << 24) + 4099, 100, 8, 4
    cent = r.standard_normal((nlist, dim)).astype(np.float32)
    books = (0.3 * r.standard_normal((M, 256, dim // M))).astype(np.float32)
    lists = r.integers(0, nlist, n).astype(np.int32)
    codes = r.integers(0, 256, (n, M)).astype(np.uint8)
    ids = np.arange(n, dtype=np.int64)[::-1].copy()
    if device:
        t = [torch.from_numpy(a).to("cuda:0") for a in (cent, books, codes, lists, ids)]
        d = amp.abi.anns_build_desc()
        d.n, d.dim, d.nlist, d.M, d.ksub = n, dim, nlist, M, 256
        d.centroids, d.codebooks, d.codes, d.list_of, d.ids = (a.data_ptr() for a in t)
        d.on_device, d.device = 1, 0
        g = amp.Index._wrap(amp.abi.anns_build_index_from_arrays(d), 0)
    else:
        g = amp.Index(cent, books, codes, lists, ids=ids, device=0)
    order = np.argsort(lists, kind="stable")
    ex = g.export()
    assert np.array_equal(ex["codes"], codes[order])
    assert np.array_equal(ex["ids"], ids[order])
    rows = np.array([0, 1, (1 << 24) - 1, 1 << 24, n - 1])
    Q = cent[lists[rows]] + books[np.arange(M)[None], codes[rows]].reshape(len(rows), dim)
    # codes repeat (2^32 of them over 17 M vectors, 100 lists): the nearest one is
    # the vector itself or another of the same list and codes
    I, D = g.search(torch.from_numpy(Q).to("cuda:0"), nlist, 1)
    got = n - 1 - I.cpu().numpy()[:, 0]
    d = ((cent[lists[got]] + books[np.arange(M)[None], codes[got]].reshape(len(rows), dim) - Q) ** 2).sum(1)
    assert (d <= 1e-4).all()
