"""qgx_quantize on both sides of the bucket counts where a bucket's threads halve, symbols against the oracle."""
import numpy as np
import pytest

import qgx_inputs as gen
from oracle import qgx_oracle as o

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bucket", [1028, 2048, 4100, 8192])
@pytest.mark.parametrize("nb", [8 * 148 - 1, 8 * 148, 8 * 148 + 1])
def test_few_and_many_buckets(bucket, nb):
    import paper_2308_09187_b200 as qgx
    ctx = qgx.qgx_create(0)
    d = nb * bucket - 5
    lev = [0.0, 0.01, 0.03, 0.2, 1.0]
    v = gen.gaussian((1, d), seed=nb, device="cuda")
    norms, sym = qgx.qgx_quantize(ctx, v, bucket, lev, qgx.QGX_NORM_L2, 9, 4)
    qgx.qgx_sync_status(ctx)
    x, n, s = v.cpu().numpy(), norms.cpu().numpy(), sym.cpu().numpy()
    for b in (0, 1, nb // 2, nb - 2, nb - 1):                # the oracle on a few buckets: whole vector, one bucket not zero
        lo, hi = b * bucket, min((b + 1) * bucket, d)
        part = np.zeros((1, hi), dtype=np.float32)
        part[0, lo:] = x[0, lo:hi]
        assert np.array_equal(o.quantize(part, bucket, lev, n[:, : b + 1], 9, 4)[0, lo:], s[0, lo:hi])
        assert abs(o.bucket_norms(part, bucket)[0, b] - n[0, b]) <= np.spacing(n[0, b])
    qgx.qgx_destroy(ctx)
