"""What a user of this library has it do, as cases that can be timed: the iteration of Algorithm 1 (and its relatives of
Sec. 3.1), one exchange of a whole or layer-wise vector, the four steps of an exchange as calls of their own, and the
refit of the levels.  Shapes, distributions and options are those of the repository's configurations (bilinear game,
affine VI, diagonal scale run, Gaussian batch, layer-wise gradients) or generic ones in between.

listed() names the cases, draw() gives more of the same ranges, prepare() makes what a program has in hand before the
call, run() is one pass through the public calls, work() what a pass cannot do without, tolerance() how far apart two
correct implementations may be."""
import math

import torch

import paper_2308_09187_b200 as qgx

CODES = {"fixed": qgx.QGX_CODE_FIXED, "huffman": qgx.QGX_CODE_HUFFMAN, "elias": qgx.QGX_CODE_ELIAS}
NORMS = {"l2": qgx.QGX_NORM_L2, "linf": qgx.QGX_NORM_LINF}


def listed():
    return [
        # a small game played for thousands of iterations: every launch counts (the bilinear configuration)
        dict(name="eg bilinear n1024 K4", kind="step", operator="bilinear", d=2048, K=4, bucket=512, sub=32, nlev=9,
             code="fixed", norm="l2", method="de", noise="additive"),
        # a mid-sized dense VI: two passes over the matrix per iteration (the affine configuration)
        dict(name="eg affine n8192 K8", kind="step", operator="affine", d=8192, K=8, bucket=4096, sub=32, nlev=17,
             code="huffman", norm="l2", method="de", noise="additive"),
        # the scale run: the largest vectors, adaptive levels, Huffman code (the diagonal configuration)
        dict(name="eg diagonal d64M K32", kind="step", operator="diagonal", d=1 << 26, K=32, bucket=16384, sub=64, nlev=17,
             code="huffman", norm="l2", method="de", noise="additive"),
        # optimistic dual averaging under random player updates: one exchange per iteration, kept symbols compared in place
        dict(name="optda relative d1M K8", kind="step", operator="diagonal", d=1000000, K=8, bucket=1024, sub=32, nlev=9,
             code="huffman", norm="l2", method="optda", noise="relative"),
        # one exchange of a large batch of Gaussian vectors (the exchange-only configuration)
        dict(name="exchange d16M K8", kind="exchange", d=1 << 24, K=8, bucket=8192, sub=64, nlev=17, code="huffman",
             norm="l2", values="gauss"),
        # one exchange of a small model's vector, bucket 1024 as in the paper's experiments: latency
        dict(name="exchange d10k K4", kind="exchange", d=10000, K=4, bucket=1024, sub=32, nlev=9, code="fixed",
             norm="l2", values="gauss"),
        # a flattened model whose parameter count is odd, largest-magnitude norms, Elias' code
        dict(name="exchange odd d1M K16", kind="exchange", d=1000003, K=16, bucket=4096, sub=32, nlev=9, code="elias",
             norm="linf", values="student"),
        # gradients of a network, tensor by tensor, each with its own levels and code (the layer-wise configuration)
        dict(name="layer-wise 16 tensors K16", kind="layers", tensors=16, first=1728, base=36864, K=16, bucket=4096, sub=32,
             nlev=9, code="huffman", norm="l2", values="student"),
        # the sending side by the separate calls: quantize, encode
        dict(name="send d4M K8", kind="send", d=1 << 22, K=8, bucket=8192, sub=64, nlev=17, code="huffman", norm="l2",
             values="gauss"),
        # the receiving side by the separate calls: decode, average
        dict(name="receive d4M K8", kind="receive", d=1 << 22, K=8, bucket=8192, sub=64, nlev=17, code="huffman", norm="l2",
             values="gauss"),
        # all four calls in a row on a small vector whose code has no sub-blocks (which the fused exchange does not take)
        dict(name="four calls d8k K4", kind="four", d=8200, K=4, bucket=512, sub=0, nlev=9, code="fixed", norm="l2",
             values="gauss"),
        # level adaptation on a large batch: histogram, fit, Huffman code
        dict(name="refit d16M K8", kind="refit", d=1 << 24, K=8, bucket=8192, sub=64, nlev=17, code="huffman", norm="l2",
             values="mixture"),
    ]


def _size(rng, lo, hi):
    """Spread over the logarithm; half of them a multiple of 64, the others as they fall."""
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    return max(64, n // 64 * 64) if rng.random() < 0.5 else n


def draw(rng):
    kind = rng.choice(["step", "step", "step", "exchange", "exchange", "layers", "send", "receive", "four", "refit"])
    c = dict(kind=kind, K=rng.choice([2, 3, 4, 8, 16]), bucket=rng.choice([512, 1024, 2048, 4096, 8192, 16384]),
             sub=rng.choice([32, 64, 128]), nlev=rng.choice([3, 5, 9, 17, 17, 32]), code=rng.choice(["fixed", "huffman", "huffman", "elias"]),
             norm=rng.choice(["l2", "l2", "l2", "linf"]))
    if kind == "step":
        c["operator"] = rng.choice(["bilinear", "affine", "diagonal", "diagonal"])
        c["method"] = rng.choice(["de", "de", "da", "optda"])
        c["noise"] = rng.choice(["additive", "additive", "relative"])
        if c["operator"] == "diagonal":
            c["K"] = rng.choice([2, 4, 8, 16, 32])
            c["d"] = _size(rng, 1000, 1 << 24)
        elif c["operator"] == "bilinear":
            c["d"], c["bucket"] = 2 * _size(rng, 64, 4096), rng.choice([256, 512, 1024])
        else:
            c["d"], c["bucket"] = _size(rng, 256, 8192), rng.choice([512, 1024, 4096])
        return c
    c["values"] = rng.choice(["gauss", "student", "mixture"])
    if kind == "exchange" or kind == "refit":
        c["d"] = _size(rng, 1000, 1 << 24)
    elif kind == "layers":
        c.update(tensors=rng.randint(3, 24), first=4 * rng.randint(8, 1000), base=_size(rng, 2000, 40000), bucket=rng.choice([1024, 4096, 8192]))
    elif kind == "send" or kind == "receive":
        c["d"] = _size(rng, 4000, 1 << 22)
    else:                                       # four: codes without sub-blocks, one bucket walked front to back
        c.update(d=_size(rng, 1000, 1 << 20), sub=rng.choice([0, 0, 32]), bucket=rng.choice([256, 512, 1024]), K=rng.choice([2, 4, 8]))
    return c


def _layer_sizes(c):
    """A few small tensors and a ladder of doubling ones, every size twice, as in a convolutional network; the vector
    ends on the last tensor's own size, whatever its remainder."""
    out, base = [], c["base"] // 4 * 4
    for j in range(c["tensors"]):
        rung = (j // 2) % 8
        out.append(c["first"] if rung == 0 else base << (rung - 1))
    out[-1] += c["base"] % 4
    return out


def _values(shape, kind, gen):
    x = torch.randn(shape, generator=gen, device="cuda")
    flat = x.view(-1)
    for lo in range(0, flat.numel(), 1 << 27):              # bounded temporaries
        part = flat[lo:lo + (1 << 27)]
        if kind == "mixture":                               # 0.9 N(0, 1) + 0.1 N(0, 100)
            part.mul_(torch.where(torch.rand(part.shape, generator=gen, device="cuda") < 0.1, 10.0, 1.0))
        elif kind == "student":                             # Student-t with three degrees of freedom
            chi = torch.zeros_like(part)
            for _ in range(3):
                chi.add_(torch.randn(part.shape, generator=gen, device="cuda").square_())
            part.div_(chi.div_(3.0).sqrt_())
    return x


def _cfg(c, seed):
    levels = [j / (c["nlev"] - 1) for j in range(c["nlev"])]
    cb = qgx.qgx_build_codebook_elias(c["nlev"], c["sub"]) if c["code"] == "elias" else qgx.qgx_build_codebook_fixed(c["nlev"], c["sub"])
    return qgx.make_quant_cfg(levels, c["bucket"], cb, seed, norm_type=NORMS[c["norm"]], code_type=CODES[c["code"]], nbins=1024)


def _operator(c, gen):
    d = c["d"]
    mode = qgx.QGX_NOISE_RELATIVE if c["noise"] == "relative" else qgx.QGX_NOISE_ADDITIVE
    if c["operator"] == "diagonal":
        return qgx.make_operator(qgx.QGX_OP_DIAGONAL, torch.rand(d, generator=gen, device="cuda") * 0.99 + 0.01, noise_model=mode)
    n = d // 2 if c["operator"] == "bilinear" else d
    g = torch.randn((n, n), generator=gen, device="cuda") * n ** -0.5
    if c["operator"] == "bilinear":
        return qgx.make_operator(qgx.QGX_OP_BILINEAR, g, noise_model=mode)
    m = ((g - g.t()) * 0.5 + 0.1 * torch.eye(n, device="cuda")).contiguous()
    return qgx.make_operator(qgx.QGX_OP_DENSE_AFFINE, m, torch.randn(n, generator=gen, device="cuda"), noise_model=mode)


def _noise(c, gen):
    if c["noise"] == "relative":                            # players of 64 coordinates, each updated with probability 1/2
        players = (c["d"] + 63) // 64
        drawn = (torch.rand((c["K"], players), generator=gen, device="cuda") < 0.5).float() * 2.0
        return drawn.repeat_interleave(64, dim=1)[:, :c["d"]].contiguous()
    return _values((c["K"], c["d"]), "mixture" if c["operator"] == "diagonal" else "gauss", gen)


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    s = dict(case=c, ctx=qgx.qgx_create(torch.cuda.current_device()), xid=3)
    K, bucket = c["K"], c["bucket"]
    adaptive = c["code"] != "fixed"
    if c["kind"] == "step":
        s["op"] = _operator(c, gen)
        s["noise"] = [_noise(c, gen) for _ in range(2 if c["method"] == "de" else 1)]
        s["st"] = qgx.EgState(torch.randn(c["d"], generator=gen, device="cuda"), K)
        s["cfg"] = _cfg(c, int(seed))
        s["mean_prev"] = torch.zeros(c["d"], device="cuda")
        qgx.qgx_eg_init(s["ctx"], s["st"])
        _step(s, qgx.QGX_REFIT_FIRST if adaptive else qgx.QGX_REFIT_NONE)      # the first iteration fits the levels
        return s
    if c["kind"] == "layers":
        s["sizes"] = _layer_sizes(c)
        parts, s["cfgs"] = [], []
        for n in s["sizes"]:
            t = _values((K, n), c["values"], gen) * 10.0 ** (-3.0 * torch.rand(1, generator=gen, device="cuda"))
            cfg = _cfg(c, int(seed))
            if adaptive:
                qgx.qgx_update_levels(s["ctx"], t, cfg, qgx.QGX_REFIT_FIRST)
            parts.append(t)
            s["cfgs"].append(cfg)
        s["v"] = torch.cat(parts, dim=1).contiguous()
        return s
    s["v"] = _values((K, c["d"]), c["values"], gen)
    s["cfg"] = _cfg(c, int(seed))
    if adaptive:
        qgx.qgx_update_levels(s["ctx"], s["v"], s["cfg"], qgx.QGX_REFIT_FIRST)
    cfg = s["cfg"]
    if c["kind"] in ("send", "receive", "four"):
        s["levels"] = cfg.level_list()
        cap = qgx.qgx_stream_capacity_words(c["d"], bucket, c["sub"], cfg.cb.maxlen)
        s["stream"] = torch.zeros((K, cap), dtype=torch.int32, device="cuda")   # kept by the program from call to call
    if c["kind"] == "receive":
        norms, sym = qgx.qgx_quantize(s["ctx"], s["v"], bucket, s["levels"], cfg.norm_type, int(seed), 3)
        _, s["bits"], _ = qgx.qgx_encode(s["ctx"], norms, sym, bucket, cfg.cb, stream=s["stream"], cap_words=s["stream"].shape[1])
    return s


def _step(s, refit):
    c = s["case"]
    if c["method"] == "de":
        qgx.qgx_eg_step(s["ctx"], s["st"], s["op"], s["noise"][0], s["noise"][1], s["cfg"], refit=refit)
    else:
        method = qgx.QGX_METHOD_OPTDA if c["method"] == "optda" else qgx.QGX_METHOD_DA
        qgx.qgx_family_step(s["ctx"], s["st"], method, s["op"], s["noise"][0], s["cfg"], refit=refit, mean_prev=s["mean_prev"])


def run(state):
    s = state
    c, ctx = s["case"], s["ctx"]
    kind, bucket = c["kind"], c["bucket"]
    if kind == "step":
        _step(s, qgx.QGX_REFIT_NONE)
        st = s["st"]
        return dict(X=st.X, Y=st.Y, Xbar=st.Xbar, Xhalf=st.Xhalf, scalars=st.scalars)
    if kind == "exchange":
        mean, bits = qgx.qgx_exchange(ctx, s["v"], s["cfg"], s["xid"])
        return dict(mean=mean, bits=bits)
    if kind == "layers":
        mean, bits = qgx.qgx_exchange_segments(ctx, s["v"], s["sizes"], s["cfgs"], s["xid"])
        return dict(mean=mean, bits=bits)
    cfg = s["cfg"]
    if kind == "refit":                                     # continues from the levels in use, as an iteration's refits do
        new = qgx.make_quant_cfg(cfg.level_list(), bucket, cfg.cb, cfg.seed, norm_type=cfg.norm_type, code_type=cfg.code_type, nbins=cfg.nbins)
        hist = qgx.qgx_update_levels(ctx, s["v"], new, qgx.QGX_REFIT_CONTINUE)
        return dict(hist=torch.tensor(hist, dtype=torch.float64), levels=torch.tensor(new.level_list()), lengths=torch.tensor(new.cb.lengths()))
    if kind == "receive":
        norms, sym = qgx.qgx_decode(ctx, s["stream"], s["bits"], c["d"], bucket, cfg.cb)
        return dict(norms=norms, sym=sym, mean=qgx.qgx_average(ctx, norms, sym, bucket, s["levels"]))
    norms, sym = qgx.qgx_quantize(ctx, s["v"], bucket, s["levels"], cfg.norm_type, cfg.seed, s["xid"])
    stream, bits, total = qgx.qgx_encode(ctx, norms, sym, bucket, cfg.cb, stream=s["stream"], cap_words=s["stream"].shape[1])
    out = dict(norms=norms, sym=sym, stream=stream, bits=bits, total=total)
    if kind == "four":
        got_norms, got_sym = qgx.qgx_decode(ctx, stream, bits, c["d"], bucket, cfg.cb)
        out["mean"] = qgx.qgx_average(ctx, got_norms, got_sym, bucket, s["levels"])
    return out


def work(case):
    """Bytes: each input once, each output once; a stream counts about half a byte per coordinate.  Operations per
    coordinate and worker: norm 2, normalize and round 5, dequantize and add 2 (the generator's integer work left out)."""
    c, K = case, case["K"]
    d = sum(_layer_sizes(c)) if c["kind"] == "layers" else c["d"]
    v = K * d
    if c["kind"] == "step":
        exchanges = 2 if c["method"] == "de" else 1
        n = d // 2 if c["operator"] == "bilinear" else d
        mat = {"bilinear": n * n, "affine": d * d, "diagonal": d}[c["operator"]]
        noise = 4.0 * v
        state = 4.0 * d * (3 + 4)                           # X, Y, Xbar and the anchor in; X, Y, Xbar, Xhalf out
        ops = 2.0 * mat * (2 if c["operator"] == "bilinear" else 1)
        return {"bytes": exchanges * (noise + 0.5 * v) + 4.0 * mat + state, "flops": exchanges * (9.0 * v + ops) + 8.0 * d}
    if c["kind"] in ("exchange", "layers"):
        return {"bytes": 4.0 * v + 0.5 * v + 4.0 * d, "flops": 9.0 * v}
    if c["kind"] == "refit":
        return {"bytes": 4.0 * v + 8.0 * 1024, "flops": 4.0 * v}
    if c["kind"] == "send":
        return {"bytes": 4.0 * v + 1.0 * v + 0.5 * v, "flops": 7.0 * v}
    if c["kind"] == "receive":
        return {"bytes": 0.5 * v + 1.0 * v + 4.0 * d, "flops": 2.0 * v}
    return {"bytes": 4.0 * v + 1.0 * v + 0.5 * v + 4.0 * d, "flops": 9.0 * v}


def tolerance(case):
    """32-bit data with 64-bit sums: a norm may be rounded the other way when its sum is taken in another order, and a
    coordinate that sits on the edge of its variate may then fall to the neighbouring level."""
    if case["kind"] == "refit":
        return {"rel": 1e-6}
    return {"rel": 1e-5, "differ": 1e-5}
