"""The separate calls at the sizes where their kernels branch: symbols that can be loaded eight, four or one at a time,
several buckets per warp and several warps per bucket, codes without sub-blocks, more buckets than one turn of the offset
scan, capacities below the worst case -- against the oracle."""
import numpy as np
import pytest
import torch

import qgx_inputs as gen
from oracle import qgx_oracle as o

pytestmark = pytest.mark.gpu

CASES = [
    # K, d, bucket, nlev, subblock
    (1, 5, 4, 2, 0),
    (3, 1003, 256, 9, 32),                  # one symbol at a time, 8 sub-blocks: four buckets per warp
    (2, 4100, 512, 17, 128),                # four at a time
    (5, 4808, 1024, 9, 0),                  # eight at a time, no sub-blocks
    (4, 16 * 500, 500, 5, 100),             # a layout that only the three-kernel encoder takes
    (2, 3 * 8192 + 4112, 8192, 32, 64),     # four warps per bucket
    (3, 16384 + 16368, 16384, 17, 32),
    (2, 4 * 5000, 4, 3, 0),                 # 5000 buckets: the scan's second turn
]


@pytest.mark.parametrize("K,d,bucket,nlev,sub", CASES)
@pytest.mark.parametrize("roomy", [True, False])
def test_steps_match_oracle(K, d, bucket, nlev, sub, roomy):
    import paper_2308_09187_b200 as qgx
    ctx = qgx.qgx_create(0)
    try:
        rng = np.random.default_rng(d + nlev)
        v = gen.gaussian_mixture((K, d), seed=d, device="cuda")
        v[0, : min(d, bucket)] = 0.0
        lev = np.r_[0.0, np.sort(rng.uniform(0.001, 0.5, size=nlev - 2)), 1.0].astype(np.float32)
        cb = qgx.qgx_build_codebook_huffman(list(rng.dirichlet(np.ones(nlev))), sub)
        cbo = o.codebook_from(cb.lengths(), cb.codes(), subblock=sub)
        norms, sym = qgx.qgx_quantize(ctx, v, bucket, lev, qgx.QGX_NORM_L2, 5, 2)
        qgx.qgx_sync_status(ctx)
        n = norms.cpu().numpy()
        assert np.all(np.abs(n - o.bucket_norms(v.cpu().numpy(), bucket)) <= np.spacing(n))
        s_ref = o.quantize(v.cpu().numpy(), bucket, lev, n, 5, 2)
        assert np.array_equal(sym.cpu().numpy(), s_ref)
        half = torch.full_like(norms, float(n.max()) * 0.25)         # supplied norms below the coordinates
        _, sym2 = qgx.qgx_quantize(ctx, v, bucket, lev, qgx.QGX_NORM_L2, 5, 2, flags=qgx.QGX_NORMS_SUPPLIED, norms=half)
        qgx.qgx_sync_status(ctx)
        assert np.array_equal(sym2.cpu().numpy(), o.quantize(v.cpu().numpy(), bucket, lev, half.cpu().numpy(), 5, 2))
        st_ref, bb_ref, tot_ref = o.encode(n, s_ref, bucket, cbo)
        used = ((bb_ref.astype(np.int64) + 31) // 32).sum(axis=1)
        cap = None if roomy else int(used.max())                     # just enough
        stream, bits, total = qgx.qgx_encode(ctx, norms, sym, bucket, cb, cap_words=cap)
        qgx.qgx_sync_status(ctx)
        assert np.array_equal(bits.cpu().numpy().view(np.uint32), bb_ref)
        assert np.array_equal(total.cpu().numpy().astype(np.uint64), tot_ref)
        got = stream.cpu().numpy().view(np.uint32)
        for k in range(K):
            assert np.array_equal(got[k, : used[k]], st_ref[k, : used[k]]) and not got[k, used[k]:].any()
        norms2, sym3 = qgx.qgx_decode(ctx, stream, bits, d, bucket, cb)
        qgx.qgx_sync_status(ctx)
        assert torch.equal(norms2, norms) and torch.equal(sym3, sym)
        mean = qgx.qgx_average(ctx, norms, sym, bucket, lev)
        qgx.qgx_sync_status(ctx)
        assert np.array_equal(mean.cpu().numpy(), o.average(n, s_ref, bucket, lev))
        if used.max() > 1:                                           # one word too few: nothing is written for that worker
            tight = torch.zeros((K, int(used.max()) - 1), dtype=torch.int32, device="cuda")
            qgx.qgx_encode(ctx, norms, sym, bucket, cb, cap_words=tight.shape[1], stream=tight)
            assert qgx.qgx_sync_status(ctx, check=False) == qgx.QGX_ERR_CAPACITY
            assert not tight[int(np.argmax(used))].any()
        if nlev < 32:
            sym[K - 1, d - 1] = 31                                   # no level of this code
            qgx.qgx_encode(ctx, norms, sym, bucket, cb)
            assert qgx.qgx_sync_status(ctx, check=False) == qgx.QGX_ERR_CORRUPT
            qgx.qgx_average(ctx, norms, sym, bucket, lev)
            assert qgx.qgx_sync_status(ctx, check=False) == qgx.QGX_ERR_CORRUPT
    finally:
        qgx.qgx_destroy(ctx)


@pytest.mark.parametrize("K,d,bucket", [(2, 37 * 64, 64), (1, 148 * 16 * 32 * 4, 4), (1, 148 * 16 * 16 * 4 + 4, 4), (3, 148 * 16 * 4 * 16 + 13, 16)])
def test_decode_without_sub_blocks_spreads_its_walks(K, d, bucket):
    """One walk per bucket, from one to thirty-two buckets in a warp: on both sides of the counts where that changes."""
    import paper_2308_09187_b200 as qgx
    ctx = qgx.qgx_create(0)
    v = torch.randn((K, d), device="cuda", generator=torch.Generator("cuda").manual_seed(d))
    cb = qgx.qgx_build_codebook_elias(9, 0)
    norms, sym = qgx.qgx_quantize(ctx, v, bucket, [j / 8 for j in range(9)], qgx.QGX_NORM_L2, 5, 1)
    stream, bits, _ = qgx.qgx_encode(ctx, norms, sym, bucket, cb)
    got_norms, got_sym = qgx.qgx_decode(ctx, stream, bits, d, bucket, cb)
    qgx.qgx_sync_status(ctx)
    assert torch.equal(got_norms, norms) and torch.equal(got_sym, sym)
    qgx.qgx_destroy(ctx)


@pytest.mark.parametrize("bucket", [4, 256, 260, 512, 516, 768, 1024, 1028, 2048])
@pytest.mark.parametrize("nb", [1, 147, 2 * 148 + 1, 9 * 148 + 5])
def test_quantize_buckets_side_by_side(bucket, nb):
    """Buckets of one to eight warps, one to eight of them in a CTA, with warps left over and not: on both sides of the
    counts where that changes.  The last bucket of every worker is short, one bucket is zero, one not finite."""
    import paper_2308_09187_b200 as qgx
    K, d = (1, nb * bucket - 3) if nb % 3 else (3, nb // 3 * bucket - 3)
    nb = o.nbuckets(d, bucket)
    ctx = qgx.qgx_create(0)
    v = torch.randn((K, d), device="cuda", generator=torch.Generator("cuda").manual_seed(d))
    v[K - 1, : min(bucket, d)] = 0.0
    lev = [0.0, 0.01, 0.02, 0.1, 0.3, 0.6, 1.0]
    for norm_type in (qgx.QGX_NORM_L2, qgx.QGX_NORM_LINF):
        norms, sym = qgx.qgx_quantize(ctx, v, bucket, lev, norm_type, 5, 2)
        qgx.qgx_sync_status(ctx)
        n, x = norms.cpu().numpy(), v.cpu().numpy()
        assert np.all(np.abs(n - o.bucket_norms(x, bucket, norm_type)) <= np.spacing(n))
        assert np.array_equal(sym.cpu().numpy(), o.quantize(x, bucket, lev, n, 5, 2))
    v[0, d - 1] = float("inf")
    _, sym2 = qgx.qgx_quantize(ctx, v, bucket, lev, qgx.QGX_NORM_LINF, 5, 2)
    assert qgx.qgx_sync_status(ctx, check=False) == qgx.QGX_ERR_NONFINITE
    last = (nb - 1) * bucket
    assert not sym2[0, last:].any() and torch.equal(sym2[0, :last], sym[0, :last]) and torch.equal(sym2[1:], sym[1:])
    qgx.qgx_destroy(ctx)


@pytest.mark.parametrize("lengths", [[1, 1], list(range(1, 13)) + [12], [5] * 32, [1] + [6] * 31, [2, 7, 7] + [3] * 5, [12] * 8])
@pytest.mark.parametrize("sub", [0, 32])
def test_decoder_table_of_every_length(lengths, sub):
    """The decoder's table: codewords below, at and above the six bits of its first half, alone and mixed; codes that use
    all their codewords and codes that leave some over."""
    import paper_2308_09187_b200 as qgx
    nlev, K, d, bucket = len(lengths), 3, 5003, 512
    order = sorted(range(nlev), key=lambda j: (lengths[j], j))
    code, words, prev = 0, [0] * nlev, lengths[order[0]]
    for j in order:                                                  # canonical: consecutive codewords, shorter ones first
        code <<= lengths[j] - prev
        words[j], prev, code = code, lengths[j], code + 1
    cb = qgx.qgx_build_codebook_fixed(nlev, sub)
    for j in range(nlev):
        cb.len[j], cb.code[j] = lengths[j], words[j]
    cb.maxlen = max(lengths)
    rng = np.random.default_rng(nlev)
    s = rng.integers(0, nlev, size=(K, d)).astype(np.uint8)
    s |= (rng.integers(0, 2, size=s.shape).astype(np.uint8) << 7) * (s > 0)
    n = rng.uniform(0.5, 2.0, size=(K, o.nbuckets(d, bucket))).astype(np.float32)
    cbo = o.codebook_from(cb.lengths(), cb.codes(), subblock=sub)
    st_ref, bb_ref, _ = o.encode(n, s, bucket, cbo)
    ctx = qgx.qgx_create(0)
    stream, bits = torch.from_numpy(st_ref.view(np.int32)).cuda(), torch.from_numpy(bb_ref.view(np.int32)).cuda()
    norms, sym = qgx.qgx_decode(ctx, stream, bits, d, bucket, cb)
    qgx.qgx_sync_status(ctx)
    assert np.array_equal(norms.cpu().numpy(), n) and np.array_equal(sym.cpu().numpy(), s)
    qgx.qgx_destroy(ctx)
