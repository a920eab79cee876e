"""Buckets of 128 coordinates: a CTA of the one-launch exchange then has a single warp, which has to bring in every table
that larger CTAs fill with one element per thread."""
import numpy as np
import pytest
import torch

import qgx_inputs as gen
from oracle import qgx_oracle as o

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,d,nlev,sub", [(1, 128, 9, 32), (2, 300, 32, 64), (16, 128 * 20 + 5, 17, 32)])
def test_one_warp_buckets_match_oracle(K, d, nlev, sub):
    import paper_2308_09187_b200 as qgx
    bucket = 128
    ctx = qgx.qgx_create(0)
    rng = np.random.default_rng(d)
    v = gen.gaussian_mixture((K, d), seed=d, device="cuda")              # both signs
    lev = np.r_[0.0, np.sort(rng.uniform(0.001, 0.5, size=nlev - 2)), 1.0].astype(np.float32)
    cb = qgx.qgx_build_codebook_huffman(list(rng.dirichlet(np.ones(nlev))), sub)
    cfg = qgx.make_quant_cfg(lev, bucket, cb, 9)
    mean, total = qgx.qgx_exchange(ctx, v, cfg, 4)
    qgx.qgx_sync_status(ctx)
    stream, bbits, _ = qgx.exchange_stream_tensors(ctx, 0, K, o.nbuckets(d, bucket))
    norms, _ = qgx.qgx_quantize(ctx, v, bucket, lev, qgx.QGX_NORM_L2, 9, 4)
    qgx.qgx_sync_status(ctx)
    n = norms.cpu().numpy()
    s_ref = o.quantize(v.cpu().numpy(), bucket, lev, n, 9, 4)
    st_ref, bb_ref, tot_ref = o.encode(n, s_ref, bucket, o.codebook_from(cb.lengths(), cb.codes(), subblock=sub))
    assert np.array_equal(bbits.cpu().numpy().view(np.uint32), bb_ref) and np.array_equal(total.cpu().numpy().astype(np.uint64), tot_ref)
    used, got = ((bb_ref.astype(np.int64) + 31) // 32).sum(axis=1), stream.cpu().numpy().view(np.uint32)
    for k in range(K):
        assert np.array_equal(got[k, : used[k]], st_ref[k, : used[k]])
    assert np.array_equal(mean.cpu().numpy(), o.average(n, s_ref, bucket, lev))
    qgx.qgx_destroy(ctx)
