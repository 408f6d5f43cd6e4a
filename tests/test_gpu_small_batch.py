"""Paths that only small or only large batches take: several blocks a query,
the one-block-per-query coarse selection, a warp per pair for the MLP, and the
FP32 coarse stage through the tensor cores. Results equal the oracle's.
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


def index(amp, dim, M, nlist, n, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    cent = r.standard_normal((nlist, dim)).astype(np.float32)
    books = (0.3 * r.standard_normal((M, 256, dim // M))).astype(np.float32)
    lo = r.integers(0, nlist, n).astype(np.int32)
    codes = r.integers(0, 256, (n, M)).astype(np.uint8)
    g = amp.Index(cent, books, codes, lo, device=0)
    return r, g, ivfpq.Index(cent, books, codes, lo)


@pytest.mark.parametrize("dim,M,nlist,n", [(32, 8, 5, 700), (50, 10, 300, 4000), (96, 48, 40, 3000)])
@pytest.mark.parametrize("nq,k", [(1, 1), (2, 32), (37, 10), (64, 7), (90, 10)])
def test_small_batches(amp, dim, M, nlist, n, nq, k):
    r, g, o = index(amp, dim, M, nlist, n, dim + nq)
    nprobe = min(nlist, 33)
    Q = (o.centroids[r.integers(0, nlist, nq)] + 0.5 * r.standard_normal((nq, dim))).astype(np.float32)
    npq = r.integers(0, nprobe + 1, nq).astype(np.int32)
    kpq = r.integers(0, k + 1, nq).astype(np.int32)
    bits = r.choice(np.array([0, 4, 6, 8, 12, 16], np.uint8), size=(nq, nprobe))
    try:
        for pol, b in ((amp.policy("plain"), 0), (amp.policy("fixed", bits=8), 8), (amp.policy("fixed", bits=16), 16),
                       (amp.policy("explicit", pair_bits=cuda(bits)), bits)):
            for kw in ({}, dict(nprobe_per_q=npq, k_per_q=kpq)):
                ids, dists = g.search(cuda(Q), nprobe, k, pol, **{f: cuda(v) for f, v in kw.items()})
                ri, rd = ivfpq.search(o, Q, nprobe, k, bits=b, **kw)
                np.testing.assert_array_equal(ids.cpu().numpy(), ri)
                np.testing.assert_array_equal(dists.cpu().numpy(), rd)
    finally:
        g.close()


@pytest.mark.parametrize("nlist", [3, 31, 600, 9000])
def test_small_coarse_selection(amp, nlist):
    """One block per query, ties in distance (repeated centroids) and nprobe up to 128."""
    r = np.random.Generator(np.random.PCG64(nlist))
    cent = r.integers(-3, 4, (nlist, 8)).astype(np.float32)   # small integers: many equal distances
    g = amp.Index(cent, r.standard_normal((2, 256, 4)).astype(np.float32), r.integers(0, 256, (nlist, 2)).astype(np.uint8),
                  np.arange(nlist, dtype=np.int32), device=0)
    Q = r.integers(-3, 4, (9, 8)).astype(np.float32)
    try:
        for nprobe in sorted({1, min(nlist, 33), min(nlist, 128)}):
            rp, rd = ivfpq.locate(ivfpq.coarse_d2_fp32(Q, cent), nprobe)
            p, pd = g.locate(cuda(Q), nprobe)
            np.testing.assert_array_equal(p.cpu().numpy(), rp)
            np.testing.assert_array_equal(pd.cpu().numpy(), rd)
    finally:
        g.close()


@pytest.mark.parametrize("nq", [3, 700])
def test_mlp_widths_small_and_large(amp, nq):
    """A warp per pair (small batches) and a thread per pair choose the same widths."""
    r, g, o = index(amp, 32, 8, 60, 6000, 4)
    nprobe = 30
    p = {f: r.uniform(-1, 1, s).astype(np.float32) for f, s in amp._PRED_SHAPES.items()}
    p["inv_std"] = np.abs(p["inv_std"]) + 0.1
    g.set_predictor(p)
    Q = (o.centroids[r.integers(0, 60, nq)] + 0.5 * r.standard_normal((nq, 32))).astype(np.float32)
    from oracle import predictor
    try:
        for tau in (0.0, 0.4, -0.7):
            g.search(cuda(Q), nprobe, 10, amp.policy("mlp", margin=tau))
            torch.cuda.synchronize()
            probes, pd = ivfpq.locate(ivfpq.coarse_d2_fp32(Q, o.centroids), nprobe)
            F = predictor.features(pd, probes, o.radius, o.sizes).reshape(-1, 5)
            w16 = predictor.to_fp16({k: p[k] for k in ("W1", "b1", "W2", "b2", "W3", "b3")})
            z = predictor.mlp_logits16(w16, predictor.normalise(F, p["mean"], p["inv_std"]))
            want = predictor.decide_bits(z, tau).reshape(nq, nprobe)
            np.testing.assert_array_equal(g.tap(amp.abi.TAP_BITS, (nq, nprobe), np.uint8), want)
    finally:
        g.close()


@pytest.mark.parametrize("dim,nlist,nq", [(48, 12000, 600), (130, 2500, 1000), (96, 8192, 400)])
def test_fp32_coarse_stage_through_the_tensor_cores(amp, dim, nlist, nq):
    """Large enough that the FP32 coarse stage takes the FP16 GEMM and the exact re-rank."""
    r, g, o = index(amp, dim, dim // 2, nlist, nlist, 8)
    Q = (o.centroids[r.integers(0, nlist, nq)] + 0.7 * r.standard_normal((nq, dim))).astype(np.float32)
    npq = r.integers(0, 101, nq).astype(np.int32)
    try:
        D2 = ivfpq.coarse_d2_fp32(Q, o.centroids)
        for nprobe, kw in ((1, {}), (100, {}), (100, dict(nprobe_per_q=npq))):
            rp, rd = (a.copy() for a in ivfpq.locate(D2, nprobe))
            if kw:
                out = np.arange(nprobe)[None, :] >= np.minimum(npq, nprobe)[:, None]
                rp[out], rd[out] = -1, np.inf
            p, pd = g.locate(cuda(Q), nprobe, **{f: cuda(v) for f, v in kw.items()})
            np.testing.assert_array_equal(p.cpu().numpy(), rp)
            np.testing.assert_array_equal(pd.cpu().numpy(), rd)
        with pytest.raises(amp.AnnsError):  # not a tensor-core CL to the caller
            g.tap(amp.abi.TAP_COARSE_CANDIDATES, (nq,), np.int32)
    finally:
        g.close()


@pytest.mark.parametrize("nlist", [17, 32, 33, 100, 128, 129, 255, 300])
@pytest.mark.parametrize("cl", ["bf16", "fp8"])
def test_short_rows_of_the_tensor_core_coarse_stage(amp, nlist, cl):
    """Every list a candidate up to 32 lists, one warp's selection up to 128, the
    block's beyond: the FP32 rule's probes and distances, ties and a repeated centroid included."""
    r = np.random.Generator(np.random.PCG64(nlist))
    C = r.standard_normal((nlist, 24)).astype(np.float32)
    C[nlist // 2] = C[1]
    Q = np.concatenate([C[:2], r.standard_normal((75, 24)).astype(np.float32), 50 * C[3:4]])
    books = r.standard_normal((4, 256, 6)).astype(np.float32)
    g = amp.Index(C, books, r.integers(0, 256, (nlist, 4)).astype(np.uint8), np.arange(nlist, dtype=np.int32), device=0)
    for nprobe in (1, 16, min(nlist, 128)):
        rp, rd = ivfpq.locate(ivfpq.coarse_d2_fp32(Q, C), nprobe)
        p, d = g.locate(torch.from_numpy(Q).to("cuda:0"), nprobe, cl=cl)
        np.testing.assert_array_equal(p.cpu().numpy(), rp)
        np.testing.assert_array_equal(d.cpu().numpy(), rd)
    g.close()
