"""The histogram where its fast bins end: bin counts that are no multiple of four, one bin, the largest count, buckets whose
norm makes nbins / norm subnormal or infinite, an all-zero bucket, and every number of quads per thread."""
import numpy as np
import pytest
import torch

from oracle import qgx_oracle as o

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bucket", [256, 1024, 4096, 16384])
@pytest.mark.parametrize("nbins", [1, 3, 30, 1023, 4096])
def test_histogram_edges(bucket, nbins):
    import paper_2308_09187_b200 as qgx
    K, d = 3, 5 * bucket + 12
    v = np.random.default_rng(nbins).standard_normal((K, d)).astype(np.float32)
    v[0, :bucket] *= np.float32(1e-39)                       # nbins / norm overflows
    v[1, :bucket] *= np.float32(3e37)                        # nbins / norm is subnormal for few bins
    v[2, :bucket] = 0.0
    v[2, bucket:2 * bucket] = 0.0
    v[2, bucket + 7] = -4.0                                  # one coordinate is the norm
    ctx = qgx.qgx_create(0)
    got = qgx.qgx_histogram(ctx, torch.from_numpy(v).cuda(), bucket, nbins, norm_type=qgx.QGX_NORM_LINF, weighted=False)
    qgx.qgx_sync_status(ctx)
    assert np.array_equal(got.cpu().numpy(), o.histogram(v, bucket, nbins, o.LINF, False))
    qgx.qgx_destroy(ctx)
