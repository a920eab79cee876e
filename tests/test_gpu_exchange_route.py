"""Which exchanges go out in one launch: shapes on both sides of the rule, where the two ways' times were measured apart.
Both ways give the same mean and bits."""
import numpy as np
import pytest
import torch

import qgx_inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,nb,bucket,nlev,one_launch", [
    (4, 10, 1024, 9, True),
    (16, 9, 4096, 9, True),
    (8, 27, 8192, 9, True),
    (12, 6, 16384, 9, True),               # as many clusters of twelve as are resident at a time ...
    (12, 9, 16384, 9, False),              # ... and more
    (16, 129, 512, 17, False),             # small buckets, large tables in every CTA
    (2, 296 * 14, 128, 17, False),
])
def test_one_launch_where_it_is_the_faster_way(K, nb, bucket, nlev, one_launch):
    import paper_2308_09187_b200 as qgx
    d = nb * bucket - 4
    v = gen.gaussian((K, d), seed=nb, device="cuda")
    if nlev == 9:
        lev, cb = np.linspace(0, 1, 9), qgx.qgx_build_codebook_fixed(9, 32)
    else:                                  # crowded levels and codewords of up to twelve bits
        lev = np.r_[0.0, 0.0005 * 1.55 ** np.arange(15), 1.0]
        cb = qgx.qgx_build_codebook_huffman([2.0 ** -(j + 1) for j in range(17)], 32)
    cfg = qgx.make_quant_cfg(lev, bucket, cb, 9)
    ctx, large = qgx.qgx_create(0), qgx.qgx_create(0)
    qgx.qgx_set_encode_path(large, qgx.QGX_ENCODE_REGISTERS)
    want = qgx.qgx_exchange(large, v, cfg, 4)
    qgx.qgx_exchange(ctx, v, cfg, 4)       # the tables are built
    before = qgx.qgx_launch_count(ctx)
    got = qgx.qgx_exchange(ctx, v, cfg, 4)
    assert (qgx.qgx_launch_count(ctx) - before == 1) == one_launch
    qgx.qgx_sync_status(ctx)
    qgx.qgx_sync_status(large)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    qgx.qgx_destroy(ctx)
    qgx.qgx_destroy(large)
