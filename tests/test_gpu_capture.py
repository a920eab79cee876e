"""The separate calls in a CUDA stream capture: what a launch needs of its level table and code travels with the launch, so
nothing is allocated while a capture runs, and a replay still uses the tables that were recorded, whatever tables other
calls on the context have used in between."""
import numpy as np
import pytest
import torch

import qgx_inputs as gen
from oracle import qgx_oracle as o

pytestmark = pytest.mark.gpu


def _levels(rng, nlev):
    return np.r_[0.0, np.sort(rng.uniform(0.001, 0.4, size=nlev - 2)), 1.0].astype(np.float32)


@pytest.mark.parametrize("K,d,bucket,nlev,sub", [(2, 3001, 512, 9, 64), (3, 2 * 8192 + 4, 8192, 32, 128)])
def test_recorded_quantize_and_encode_keep_their_levels(K, d, bucket, nlev, sub):
    import paper_2308_09187_b200 as qgx
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx, warm = qgx.qgx_create(0), qgx.qgx_create(0)
        rng = np.random.default_rng(d)
        v = gen.gaussian_mixture((K, d), seed=d, device="cuda")
        lev, cb, nb = _levels(rng, nlev), qgx.qgx_build_codebook_fixed(nlev, sub), o.nbuckets(d, bucket)
        norms, sym = torch.empty((K, nb), device="cuda"), torch.empty((K, d), dtype=torch.uint8, device="cuda")
        cap = qgx.qgx_stream_capacity_words(d, bucket, sub, cb.maxlen)
        out = torch.zeros((K, cap), dtype=torch.int32, device="cuda")
        bits, total = torch.empty((K, nb), dtype=torch.int32, device="cuda"), torch.empty((K,), dtype=torch.int64, device="cuda")
        # the module is loaded and the encoder's scratch address known; `ctx` itself has not quantized yet
        qgx.qgx_quantize(warm, v, bucket, _levels(rng, nlev), qgx.QGX_NORM_L2, 5, 2, norms=norms, sym=sym)
        qgx.qgx_encode_noalloc(warm, norms, sym, bucket, cb, out, bits, total)
        qgx.qgx_sync_status(warm)
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        try:
            qgx.qgx_quantize(ctx, v, bucket, lev, qgx.QGX_NORM_L2, 5, 2, norms=norms, sym=sym)
            qgx.qgx_encode_noalloc(ctx, norms, sym, bucket, cb, out, bits, total)
        finally:
            graph.capture_end()
        for _ in range(24):                                  # more level tables than a context keeps
            qgx.qgx_quantize(ctx, v, bucket, _levels(rng, nlev), qgx.QGX_NORM_L2, 5, 2)
        v.copy_(gen.gaussian_mixture((K, d), seed=d + 1, device="cuda"))
        out.zero_()
        graph.replay()
        qgx.qgx_sync_status(ctx)
        n = norms.cpu().numpy()
        s_ref = o.quantize(v.cpu().numpy(), bucket, lev, n, 5, 2)
        assert np.array_equal(sym.cpu().numpy(), s_ref)
        st_ref, bb_ref, tot_ref = o.encode(n, s_ref, bucket, o.codebook_from(cb.lengths(), cb.codes(), subblock=sub))
        assert np.array_equal(bits.cpu().numpy().view(np.uint32), bb_ref) and np.array_equal(total.cpu().numpy().astype(np.uint64), tot_ref)
        used = ((bb_ref.astype(np.int64) + 31) // 32).sum(axis=1)
        got = out.cpu().numpy().view(np.uint32)
        for k in range(K):
            assert np.array_equal(got[k, : used[k]], st_ref[k, : used[k]])
        del graph
        qgx.qgx_destroy(ctx)
        qgx.qgx_destroy(warm)


@pytest.mark.parametrize("K,d,bucket,nlev,sub", [(2, 3001, 512, 9, 0), (3, 2 * 8192 + 4, 8192, 32, 128)])
def test_recorded_decode_keeps_its_code(K, d, bucket, nlev, sub):
    import paper_2308_09187_b200 as qgx
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = qgx.qgx_create(0)
        rng = np.random.default_rng(d)
        v = gen.gaussian_mixture((K, d), seed=d, device="cuda")
        codes = [qgx.qgx_build_codebook_huffman(list(rng.dirichlet(np.ones(nlev) * 0.5)), sub) for _ in range(24)]
        norms, sym = qgx.qgx_quantize(ctx, v, bucket, _levels(rng, nlev), qgx.QGX_NORM_L2, 5, 2)
        sent = [qgx.qgx_encode(ctx, norms, sym, bucket, cb)[:2] for cb in codes]
        got_norms, got_sym = torch.empty_like(norms), torch.empty_like(sym)
        qgx.qgx_decode(ctx, *sent[1], d, bucket, codes[1], norms=got_norms, sym=got_sym)   # the workspace has its size
        qgx.qgx_sync_status(ctx)
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        try:
            qgx.qgx_decode(ctx, *sent[0], d, bucket, codes[0], norms=got_norms, sym=got_sym)
        finally:
            graph.capture_end()
        for at, cb in zip(sent[1:], codes[1:]):
            _, other = qgx.qgx_decode(ctx, *at, d, bucket, cb)
            assert torch.equal(other, sym)
        got_norms.zero_()
        got_sym.zero_()
        graph.replay()
        qgx.qgx_sync_status(ctx)
        assert torch.equal(got_norms, norms) and torch.equal(got_sym, sym)
        del graph
        qgx.qgx_destroy(ctx)
