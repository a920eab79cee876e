"""The pipelined encode kernel at the sizes where it can go wrong: one lane, one chunk and one unit more or less, the rings
of its stages and images turning over, rows off the 16-byte grid, every way of cutting a bucket into chunks -- streams and
means bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import qgx_inputs as gen
from oracle import qgx_oracle as o

pytestmark = pytest.mark.gpu

CASES = [
    # K, d, bucket, nlev, subblock, huffman, norm
    (1, 1, 1024, 2, 32, False, "l2"),                       # a single coordinate
    (3, 1023, 1024, 9, 32, True, "l2"),                     # a lane that is not full
    (2, 1025, 1024, 9, 64, True, "linf"),                   # one coordinate in the second bucket
    (5, 4096 + 33, 2048, 17, 128, True, "l2"),              # an odd number of sub-blocks in the tail, odd rows
    (4, 3 * 4096 + 1024, 4096, 9, 32, False, "l2"),         # the tail is one whole chunk
    (2, 2 * 8192 + 5121, 8192, 32, 64, False, "linf"),      # 13-bit symbols' worth of room, several chunks in the tail
    (3, 16384 + 16383, 16384, 17, 128, True, "l2"),
    (2, 1200 * 1024 + 1, 1024, 5, 32, True, "l2"),          # every CTA turns its rings over, odd rows
    (7, 60 * 16384 + 8190, 16384, 17, 64, True, "l2"),
]


@pytest.mark.parametrize("K,d,bucket,nlev,sub,huff,norm", CASES)
def test_pipeline_streams_match_oracle(K, d, bucket, nlev, sub, huff, norm):
    import paper_2308_09187_b200 as qgx
    ctx = qgx.qgx_create(0)
    try:
        qgx.qgx_set_encode_path(ctx, qgx.QGX_ENCODE_STAGED)
        rng = np.random.default_rng(d)
        v = gen.gaussian_mixture((K, d), seed=d + 7, device="cuda")
        v[K - 1, : min(d, bucket)] = 0.0                     # a bucket without a norm
        lev = np.r_[0.0, np.sort(rng.uniform(0.001, 0.2, size=nlev - 2)), 1.0].astype(np.float32)
        cb = qgx.qgx_build_codebook_huffman(list(rng.dirichlet(np.ones(nlev) * 0.4)), sub) if huff else qgx.qgx_build_codebook_fixed(nlev, sub)
        cbo = o.codebook_from(cb.lengths(), cb.codes(), subblock=sub)
        kind = qgx.QGX_NORM_L2 if norm == "l2" else qgx.QGX_NORM_LINF
        cfg = qgx.make_quant_cfg(lev, bucket, cb, 31, norm_type=kind)
        nb = o.nbuckets(d, bucket)
        mean, total = qgx.qgx_exchange(ctx, v, cfg, 12, slot=0)
        qgx.qgx_sync_status(ctx)
        stream, bbits, _ = qgx.exchange_stream_tensors(ctx, 0, K, nb)
        norms, sym = qgx.qgx_quantize(ctx, v, bucket, lev, kind, 31, 12)
        qgx.qgx_sync_status(ctx)
        n_gpu = norms.cpu().numpy()
        s_ref = o.quantize(v.cpu().numpy(), bucket, lev, n_gpu, 31, 12)
        st_ref, bb_ref, tot_ref = o.encode(n_gpu, s_ref, bucket, cbo)
        assert np.array_equal(sym.cpu().numpy(), s_ref)
        assert np.array_equal(bbits.cpu().numpy().view(np.uint32), bb_ref)
        assert np.array_equal(total.cpu().numpy().astype(np.uint64), tot_ref)
        got = stream.cpu().numpy().view(np.uint32)
        used = ((bb_ref.astype(np.int64) + 31) // 32).sum(axis=1)
        for k in range(K):
            assert np.array_equal(got[k, : used[k]], st_ref[k, : used[k]])
        assert np.array_equal(mean.cpu().numpy(), o.average(n_gpu, s_ref, bucket, lev))
    finally:
        qgx.qgx_destroy(ctx)
