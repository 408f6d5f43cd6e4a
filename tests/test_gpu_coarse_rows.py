"""The re-rank's selection of the tensor-core coarse stage by row length: the
radix select of 129 to 2048 lists and the bisection beyond give the FP32 rule's
probes and distances on both sides of the line, with ties, repeated centroids,
few and many candidates (more than the split re-rank's 512), per-query nprobe
and a NaN query."""
import numpy as np
import pytest

from oracle import ivfpq

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nlist,dim", [(129, 24), (700, 30), (1024, 96), (2048, 20), (2049, 20)])
@pytest.mark.parametrize("cl", ["fp16", "fp8"])
def test_rows_around_the_radix_select(nlist, dim, cl):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_07156_gb300 as amp
    r = np.random.Generator(np.random.PCG64(nlist))
    C = r.standard_normal((nlist, dim)).astype(np.float32)
    C[nlist // 2] = C[1]
    C[2:2 + min(600, nlist // 2 - 4)] = C[2]          # equal distances: every one a candidate
    Q = np.concatenate([C[:3], r.standard_normal((60, dim)).astype(np.float32), 50 * C[3:4]])
    npq = r.integers(0, 129, len(Q)).astype(np.int32)
    g = amp.Index(C, r.standard_normal((2, 256, dim // 2)).astype(np.float32),
                  r.integers(0, 256, (nlist, 2)).astype(np.uint8), np.arange(nlist, dtype=np.int32), device=0)
    D2 = ivfpq.coarse_d2_fp32(Q, C)
    try:
        for nprobe, kw in ((1, {}), (48, {}), (128, dict(nprobe_per_q=npq))):
            rp, rd = (a.copy() for a in ivfpq.locate(D2, nprobe))
            if kw:
                out = np.arange(nprobe)[None, :] >= np.minimum(npq, nprobe)[:, None]
                rp[out], rd[out] = -1, np.inf
            p, d = g.locate(torch.from_numpy(Q).to("cuda:0"), nprobe, cl=cl,
                            **{f: torch.from_numpy(v).to("cuda:0") for f, v in kw.items()})
            np.testing.assert_array_equal(p.cpu().numpy(), rp)
            np.testing.assert_array_equal(d.cpu().numpy(), rd)
        Q[7, 2] = np.nan
        p, d = (t.cpu().numpy() for t in g.locate(torch.from_numpy(Q).to("cuda:0"), 16, cl=cl))
        assert (p[7] == -1).all() and np.isinf(d[7]).all()
        rp, rd = ivfpq.locate(D2, 16)
        keep = np.arange(len(Q)) != 7
        np.testing.assert_array_equal(p[keep], rp[keep])
        np.testing.assert_array_equal(d[keep], rd[keep])
    finally:
        g.close()


@pytest.mark.parametrize("nq,nlist,dim,nprobe", [(64, 33, 24, 8), (64, 33, 24, 9), (3, 256, 100, 8), (3, 257, 100, 8),
                                                 (3, 32, 768, 32), (40, 1300, 768, 40), (41, 1300, 768, 40), (64, 4096, 100, 16),
                                                 (65, 4096, 36, 16)])
def test_few_queries_by_the_fp32_rule(nq, nlist, dim, nprobe):
    """Both sides of the lines between the small kernels and the others: a thread or a tile for the
    distances, a block or a warp for the selection, with tied distances and per-query nprobe."""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_07156_gb300 as amp
    r = np.random.Generator(np.random.PCG64(nq + nlist))
    C = r.standard_normal((nlist, dim)).astype(np.float32)
    C[5:9] = C[4]
    Q = np.concatenate([C[3:6], r.standard_normal((nq, dim)).astype(np.float32)])[:nq]
    npq = r.integers(0, nprobe + 1, nq).astype(np.int32)
    g = amp.Index(C, r.standard_normal((2, 256, dim // 2)).astype(np.float32),
                  r.integers(0, 256, (nlist, 2)).astype(np.uint8), np.arange(nlist, dtype=np.int32), device=0)
    try:
        D2 = ivfpq.coarse_d2_fp32(Q, C)
        rp, rd = ivfpq.locate(D2, nprobe)
        p, d = g.locate(torch.from_numpy(Q).to("cuda:0"), nprobe)
        np.testing.assert_array_equal(p.cpu().numpy(), rp)
        np.testing.assert_array_equal(d.cpu().numpy(), rd)
        out = np.arange(nprobe)[None, :] >= npq[:, None]
        p, d = g.locate(torch.from_numpy(Q).to("cuda:0"), nprobe, nprobe_per_q=torch.from_numpy(npq).to("cuda:0"))
        np.testing.assert_array_equal(p.cpu().numpy(), np.where(out, -1, rp))
        np.testing.assert_array_equal(d.cpu().numpy(), np.where(out, np.inf, rd))
    finally:
        g.close()
