"""Every bounded wait between CTAs can be made to run out: buckets left unencoded on purpose and a small limit.  The call
ends by itself, QGX_ERR_TIMEOUT is latched, and the next call on the context is exact."""
import time

import numpy as np
import pytest
import torch

import qgx_inputs as gen

pytestmark = pytest.mark.gpu

LEVELS = np.linspace(0, 1, 9, dtype=np.float32)
DEFAULT_LIMIT = 1 << 22


@pytest.mark.parametrize("sub", [0, 64])
def test_one_pass_encode_wait_runs_out(sub):
    import paper_2308_09187_b200 as qgx
    ctx = qgx.qgx_create(0)
    K, d, bucket = 3, 12 * 1024 + 40, 1024
    v, cb = gen.gaussian((K, d), seed=4, device="cuda"), qgx.qgx_build_codebook_fixed(9, sub)
    norms, sym = qgx.qgx_quantize(ctx, v, bucket, LEVELS, qgx.QGX_NORM_L2, 3, 1)
    want = [t.clone() for t in qgx.qgx_encode(ctx, norms, sym, bucket, cb)]
    qgx.qgx_sync_status(ctx)
    qgx.qgx_set_wait_limit(ctx, 50)
    for skip in (2, 13):                                     # the second leaves out everything: nobody waits
        qgx.qgx_debug_skip_buckets(ctx, skip)
        qgx.qgx_encode(ctx, norms, sym, bucket, cb)
        assert qgx.qgx_sync_status(ctx, check=False) == (qgx.QGX_ERR_TIMEOUT if skip == 2 else qgx.QGX_OK)
    qgx.qgx_set_wait_limit(ctx, DEFAULT_LIMIT)
    got = qgx.qgx_encode(ctx, norms, sym, bucket, cb)
    qgx.qgx_sync_status(ctx)
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    qgx.qgx_destroy(ctx)


@pytest.mark.parametrize("K,bucket", [(3, 1024), (12, 512), (1, 128)])
def test_one_launch_exchange_wait_runs_out(K, bucket):
    import paper_2308_09187_b200 as qgx
    ctx = qgx.qgx_create(0)
    d = 12 * bucket + 40
    v = gen.gaussian((K, d), seed=4, device="cuda")
    cfg = qgx.make_quant_cfg(LEVELS, bucket, qgx.qgx_build_codebook_fixed(9, 32), 3)
    want = [t.clone() for t in qgx.qgx_exchange(ctx, v, cfg, 1)]
    qgx.qgx_sync_status(ctx)
    qgx.qgx_set_wait_limit(ctx, 50)
    qgx.qgx_debug_skip_buckets(ctx, 2)
    before = qgx.qgx_launch_count(ctx)
    qgx.qgx_exchange(ctx, v, cfg, 1)
    assert qgx.qgx_launch_count(ctx) == before + 1           # it is the one launch that waited
    assert qgx.qgx_sync_status(ctx, check=False) == qgx.QGX_ERR_TIMEOUT
    qgx.qgx_set_wait_limit(ctx, DEFAULT_LIMIT)
    for _ in range(2):                                       # the scan's words were left as they were found
        got = qgx.qgx_exchange(ctx, v, cfg, 1)
        qgx.qgx_sync_status(ctx)
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    qgx.qgx_destroy(ctx)


def test_layer_wise_exchange_waits_follow_the_context():
    """The tensors run on helper contexts, made at the first such exchange: a limit set after that holds for them too."""
    import paper_2308_09187_b200 as qgx
    ctx = qgx.qgx_create(0)
    K, bucket, sizes = 2, 1024, [8 * 1024, 700 * 1024, 3 * 1024]     # one launch, the large kernels, one launch
    v = gen.gaussian((K, sum(sizes)), seed=4, device="cuda")
    cfgs = [qgx.make_quant_cfg(LEVELS, bucket, qgx.qgx_build_codebook_fixed(9, 32), 3 + s) for s in range(len(sizes))]
    want = [t.clone() for t in qgx.qgx_exchange_segments(ctx, v, sizes, cfgs, 1)]
    qgx.qgx_sync_status(ctx)
    qgx.qgx_set_wait_limit(ctx, 50)
    qgx.qgx_debug_skip_buckets(ctx, 2)
    start = time.perf_counter()
    qgx.qgx_exchange_segments(ctx, v, sizes, cfgs, 1)
    assert qgx.qgx_sync_status(ctx, check=False) == qgx.QGX_ERR_TIMEOUT
    assert time.perf_counter() - start < 1.0                 # (with the default limit: seconds)
    qgx.qgx_set_wait_limit(ctx, DEFAULT_LIMIT)
    got = qgx.qgx_exchange_segments(ctx, v, sizes, cfgs, 1)
    qgx.qgx_sync_status(ctx)
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    qgx.qgx_destroy(ctx)


@pytest.mark.parametrize("limit", [50, 1 << 15])
def test_pipelined_encode_ends_when_many_waits_run_out(limit):
    """Every worker's first unit is missing, so the scanners' waits run out one after the other while the other warps of
    their CTAs wait for them at barriers: whichever gives up first, the launch ends soon and says so."""
    import paper_2308_09187_b200 as qgx
    ctx = qgx.qgx_create(0)
    qgx.qgx_set_encode_path(ctx, qgx.QGX_ENCODE_STAGED)
    K, bucket, d = 64, 1024, 300 * 1024 + 5
    v = gen.gaussian((K, d), seed=4, device="cuda")
    cfg = qgx.make_quant_cfg(LEVELS, bucket, qgx.qgx_build_codebook_fixed(9, 32), 3)
    want = [t.clone() for t in qgx.qgx_exchange(ctx, v, cfg, 1)]
    qgx.qgx_sync_status(ctx)
    qgx.qgx_set_wait_limit(ctx, limit)
    qgx.qgx_debug_skip_buckets(ctx, 4)
    start = time.perf_counter()
    qgx.qgx_exchange(ctx, v, cfg, 1)
    assert qgx.qgx_sync_status(ctx, check=False) == qgx.QGX_ERR_TIMEOUT
    assert time.perf_counter() - start < 2.0
    qgx.qgx_set_wait_limit(ctx, DEFAULT_LIMIT)
    got = qgx.qgx_exchange(ctx, v, cfg, 1)
    qgx.qgx_sync_status(ctx)
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    qgx.qgx_destroy(ctx)
