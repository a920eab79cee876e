"""Exchanges of different shapes one after the other on the same slot of one context, among them one whose waits run out and one
whose tables are new: sums and scan words are left zero for the next, and no kernel starts on tables that are being built."""
import numpy as np
import pytest
import torch

import qgx_inputs as gen

pytestmark = pytest.mark.gpu


def _cfg(qgx, bucket, nlev, sub, seed):
    lev = np.linspace(0, 1, nlev, dtype=np.float32) ** (1.0 + 0.01 * seed)
    return qgx.make_quant_cfg(lev, bucket, qgx.qgx_build_codebook_elias(nlev, sub), seed)


@pytest.mark.parametrize("split", ["AUTO", "NEVER"])
def test_shapes_in_turn(split):
    import paper_2308_09187_b200 as qgx
    shapes = [(8, 300000, 4096, 9, 64), (3, 70001, 1024, 17, 32), (16, 300000, 512, 9, 32), (8, 300000, 4096, 9, 64), (1, 5000, 2048, 5, 128),
              (40, 40000, 8192, 32, 64), (2, 1000000, 16384, 17, 64)]
    vs = [gen.gaussian_mixture((K, d), seed=i, device="cuda") for i, (K, d, *_) in enumerate(shapes)]

    def run(ctx, i, seed):
        K, d, bucket, nlev, sub = shapes[i]
        mean, bits = qgx.qgx_exchange(ctx, vs[i], _cfg(qgx, bucket, nlev, sub, seed), 3)
        return mean, bits

    want = {}
    for i in range(len(shapes)):
        for seed in (1, 2):
            ctx = qgx.qgx_create(0)
            qgx.qgx_set_decode_split(ctx, getattr(qgx, "QGX_SPLIT_" + split))
            want[i, seed] = [t.clone() for t in run(ctx, i, seed)]
            qgx.qgx_sync_status(ctx)
            qgx.qgx_destroy(ctx)
    ctx = qgx.qgx_create(0)
    qgx.qgx_set_decode_split(ctx, getattr(qgx, "QGX_SPLIT_" + split))
    got = {}
    for turn in range(3):
        for i in range(len(shapes)):
            got[i] = run(ctx, i, 1 + turn % 2), 1 + turn % 2
        if turn == 1:                                        # buckets left out: the waits for them run out
            torch.cuda.synchronize()
            assert qgx.qgx_sync_status(ctx, check=False) == qgx.QGX_OK
            qgx.qgx_set_wait_limit(ctx, 50)
            qgx.qgx_debug_skip_buckets(ctx, 2)
            run(ctx, 0, 1)
            assert qgx.qgx_sync_status(ctx, check=False) == qgx.QGX_ERR_TIMEOUT
            qgx.qgx_set_wait_limit(ctx, 1 << 22)
        for i, (pair, seed) in got.items():
            assert torch.equal(pair[0], want[i, seed][0]) and torch.equal(pair[1], want[i, seed][1]), (turn, i)
    assert qgx.qgx_sync_status(ctx, check=False) == qgx.QGX_OK
    qgx.qgx_destroy(ctx)
