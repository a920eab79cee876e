"""The one-launch exchange at the edges of what it takes: every way of cutting a bucket into threads, ragged tails and rows,
cluster sizes, buckets that look back, repeated calls on one context (the scan's words have to be left as they were found),
kept symbols -- against the large kernels' way, which the other tests compare with the oracle."""
import numpy as np
import pytest
import torch

import qgx_inputs as gen

pytestmark = pytest.mark.gpu

CASES = [
    # K, d, bucket, nlev, subblock, norm
    (1, 1, 128, 2, 32, "l2"),
    (3, 1001, 256, 9, 64, "l2"),
    (8, 10000, 512, 17, 128, "linf"),
    (4, 25557, 1024, 9, 32, "l2"),
    (5, 2048 * 3 + 1, 2048, 32, 64, "l2"),
    (7, 4096 * 4 + 4095, 4096, 17, 128, "l2"),
    (2, 8192 * 2 + 4, 8192, 5, 32, "linf"),
    (4, 16384 + 8200, 16384, 17, 64, "l2"),
    (16, 5 * 1024 + 12, 1024, 9, 32, "l2"),                  # more workers than a portable cluster has CTAs
    (11, 16384, 16384, 9, 128, "l2"),
    (2, 256 * 300 + 17, 256, 9, 32, "l2"),
]


@pytest.mark.parametrize("K,d,bucket,nlev,sub,norm", CASES)
def test_one_launch_matches_large_kernels(K, d, bucket, nlev, sub, norm):
    import paper_2308_09187_b200 as qgx
    small, large = qgx.qgx_create(0), qgx.qgx_create(0)
    try:
        qgx.qgx_set_encode_path(large, qgx.QGX_ENCODE_REGISTERS)
        qgx.qgx_set_decode_split(large, qgx.QGX_SPLIT_NEVER)
        for c in (small, large):
            qgx.qgx_set_keep_symbols(c, True)
        rng = np.random.default_rng(d)
        lev = np.r_[0.0, np.sort(rng.uniform(0.001, 0.4, size=nlev - 2)), 1.0].astype(np.float32)
        cb = qgx.qgx_build_codebook_huffman(list(rng.dirichlet(np.ones(nlev) * 0.4)), sub)
        cfg = qgx.make_quant_cfg(lev, bucket, cb, 9, norm_type=qgx.QGX_NORM_L2 if norm == "l2" else qgx.QGX_NORM_LINF)
        nb = (d + bucket - 1) // bucket
        for xid in (4, 5, 6):
            v = gen.gaussian_mixture((K, d), seed=d + xid, device="cuda")
            v[K - 1, : min(d, bucket)] = 0.0
            (m0, t0), (m1, t1) = (qgx.qgx_exchange(c, v, cfg, xid, slot=xid & 1) for c in (small, large))
            qgx.qgx_sync_status(small)
            qgx.qgx_sync_status(large)
            assert torch.equal(m0, m1) and torch.equal(t0, t1)
            (s0, b0, q0), (s1, b1, q1) = (qgx.exchange_stream_tensors(c, xid & 1, K, nb) for c in (small, large))
            assert torch.equal(b0, b1) and torch.equal(q0, q1)
            words = ((b0.to(torch.int64) + 31) // 32).sum(dim=1).tolist()
            for k in range(K):
                assert torch.equal(s0[k, : words[k]], s1[k, : words[k]])
            assert torch.equal(qgx.qgx_level_counts(small), qgx.qgx_level_counts(large))
            assert torch.equal(qgx.qgx_exchange_decode(small, K, d, cfg, slot=xid & 1), m1)
        v[0, d // 2] = float("nan")
        qgx.qgx_exchange(small, v, cfg, 7)
        assert qgx.qgx_sync_status(small, check=False) == qgx.QGX_ERR_NONFINITE
    finally:
        qgx.qgx_destroy(small)
        qgx.qgx_destroy(large)


@pytest.mark.parametrize("method", ["de", "da", "optda"])
def test_iterations_match_large_kernels(method):
    import paper_2308_09187_b200 as qgx
    K, n, bucket = 4, 513, 256                               # d = 1026: not a multiple of four
    g = gen.c1_bilinear(n=n, K=K, T=6, device="cuda", bucket=bucket)
    got = []
    for path in (qgx.QGX_ENCODE_AUTO, qgx.QGX_ENCODE_REGISTERS):
        ctx = qgx.qgx_create(0)
        qgx.qgx_set_encode_path(ctx, path)
        cfg = qgx.make_quant_cfg(gen.uniform_levels(9).numpy(), bucket, qgx.qgx_build_codebook_fixed(9, 32), 3)
        op, st, prev = qgx.make_operator(qgx.QGX_OP_BILINEAR, g.A), qgx.EgState(g.z0, K), torch.zeros_like(g.z0)
        qgx.qgx_eg_init(ctx, st)
        for t in range(6):
            if method == "de":
                qgx.qgx_eg_step(ctx, st, op, g.noise[t, 0], g.noise[t, 1], cfg)
            else:
                qgx.qgx_family_step(ctx, st, qgx.QGX_METHOD_DA if method == "da" else qgx.QGX_METHOD_OPTDA, op, g.noise[t, 0], cfg, mean_prev=prev)
        qgx.qgx_sync_status(ctx)
        got.append((st.X.clone(), st.Y.clone(), st.Xbar.clone(), st.scalars.clone()))
        qgx.qgx_destroy(ctx)
    for x, y in zip(got[0], got[1]):
        assert torch.allclose(x, y, rtol=1e-6, atol=1e-7)
