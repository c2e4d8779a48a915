"""The measured cases: what a program that decodes with this library has it do.

A case is a dict of plain values.  Kinds:

  step    one block step of a decoder: the block input built on the device, q new rows per
          sequence through every layer, greedy acceptance (`accept`) where tokens are compared
  tree    the same pass over a draft tree (positions and attention follow the parents)
  prompt  a prompt of n + 1 tokens: the prefill of n positions, then the first block
  attn    block-causal attention of q rows against a cache of about ctx slots
  gemm    one projection, y = x W^T, by itself
  accept  target selection, verification and commit length on given logits

The whole 7B-shaped decoder is one case; the other model cases keep its (or the 13B-shaped
decoder's) layer dimensions and LM head with a few layers, so that each takes its layers'
time and an error stays what a few layers make of it.
"""
import math
from types import SimpleNamespace

import torch

import paper_2403_18647_gb300 as sd

DIMS = {
    #        d_model heads head_dim ffn   vocab  adaptive id
    "tiny": (256, 4, 64, 688, 4104, 4096),
    "7b": (4096, 32, 128, 11008, 32016, 32011),
    "13b": (5120, 40, 128, 13824, 32016, 32011),
}
EPS, THETA = 1e-5, 1e4
# the projections of the two decoders, (K, N): QKV, O, gate + up, down, LM head
PROJ = [(4096, 12288), (4096, 4096), (4096, 22016), (11008, 4096), (4096, 32016),
        (5120, 15360), (5120, 5120), (5120, 27648), (13824, 5120), (5120, 32016)]


def listed():
    return [
        # one loop iteration of a small decoder: nothing but launches and latency
        dict(name="tiny step", kind="step", dims="tiny", layers=2, b=1, q=6, ctx=128, accept=True),
        # the whole 7B-shaped decoder, one sequence: k = 5 drafts verified after a 2048-token prompt
        dict(name="7b step", kind="step", dims="7b", layers=32, b=1, q=6, ctx=2048, accept=False),
        # the 13B-shaped decoder's layers after a 4096-token prompt
        dict(name="13b step", kind="step", dims="13b", layers=4, b=1, q=6, ctx=4096, accept=False),
        # four sequences decoded together, each at its own length
        dict(name="7b step, batch 4", kind="step", dims="7b", layers=4, b=4, q=6, ctx=1024, accept=False),
        # the tree-structured second draft step: two chains of five drafts below the root
        dict(name="7b tree step", kind="tree", dims="7b", layers=4, b=1, q=11, ctx=2048, width=2),
        # a short question: 99 prompt positions, then the first block
        dict(name="short prompt", kind="prompt", dims="7b", layers=2, n=99, q=6),
        # a whole source file: 4095 prompt positions, then the first block
        dict(name="long prompt", kind="prompt", dims="7b", layers=2, n=4095, q=6),
        # attention by itself: a short context (latency) and a long one with a wide block
        dict(name="attention, 500 slots", kind="attn", b=1, q=6, heads=32, hd=128, ctx=500),
        dict(name="attention, 16384 slots", kind="attn", b=1, q=11, heads=32, hd=128, ctx=16384),
        # the largest projection of a decode step, and one of a prompt chunk
        dict(name="projection, 6 rows", kind="gemm", M=6, K=4096, N=22016),
        dict(name="projection, 500 rows", kind="gemm", M=500, K=4096, N=12288),
        # nucleus verification of four sequences, k = 5 drafts each
        dict(name="nucleus, batch 4", kind="accept", b=4, q=6, vocab=32016, temperature=0.2, top_p=0.95, top_k=0),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "tree", "prompt", "prompt", "attn", "attn", "gemm", "gemm", "accept"])
    if kind == "step":
        dims = rng.choice(["tiny", "7b", "7b", "13b"])
        b = _log(rng, 1, 8)
        q = rng.randint(1, min(16, 64 // b))
        top = 500 if dims == "tiny" else 16384 // b
        return dict(kind=kind, dims=dims, layers=rng.randint(1, 4), b=b, q=q, ctx=_log(rng, 16, top),
                    accept=dims == "tiny")
    if kind == "tree":
        width = rng.randint(2, 5)
        return dict(kind=kind, dims=rng.choice(["7b", "13b"]), layers=rng.randint(1, 4), b=rng.randint(1, 3),
                    q=1 + width * rng.randint(1, 15 // width), ctx=_log(rng, 64, 5000), width=width)
    if kind == "prompt":
        dims = rng.choice(["7b", "7b", "13b"])
        return dict(kind=kind, dims=dims, layers=rng.randint(1, 2) if dims == "7b" else 1, n=_log(rng, 3, 4095),
                    q=rng.randint(1, 16))
    if kind == "attn":
        b = _log(rng, 1, 8)
        return dict(kind=kind, b=b, q=rng.randint(1, min(16, 64 // b)), heads=rng.choice([32, 40]),
                    hd=rng.choice([64, 128, 128]), ctx=_log(rng, 16, 32000 // b))
    if kind == "gemm":
        K, N = rng.choice(PROJ)
        if rng.random() < 0.3:
            K, N = 8 * rng.randint(32, 1000), rng.randint(100, 20000)
        return dict(kind=kind, M=_log(rng, 1, 512), K=K, N=N)
    b = _log(rng, 1, 8)
    return dict(kind="accept", b=b, q=rng.randint(1, min(16, 64 // b)), vocab=rng.choice([4104, 32016, 32016]),
                temperature=rng.choice([0.0, 0.2, 0.2, 1.0]), top_p=rng.choice([0.9, 0.95]), top_k=rng.choice([0, 0, 10, 50]))


# ---- inputs -----------------------------------------------------------------------------------


def _gen(seed, stream=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + stream)
    return g


def _normal(g, shape, std, dtype=torch.bfloat16, mean=0.0):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(mean, std, generator=g)


def _ids(g, n, upper):
    return torch.randint(0, upper, (n,), generator=g, device="cuda", dtype=torch.int32)


def _layer(case, seed, layer):
    """One layer's weights: N(0, 0.02) matrices, gains around 1."""
    d, H, hd, F, _, _ = DIMS[case["dims"]]
    g, R = _gen(seed, 10 + layer), H * hd
    w = {n: _normal(g, s, 0.02) for n, s in (("wq", (R, d)), ("wk", (R, d)), ("wv", (R, d)), ("wo", (d, R)),
                                             ("w_gate", (F, d)), ("w_up", (F, d)), ("w_down", (d, F)))}
    return dict(w, attn_norm=_normal(g, (d,), 0.1, mean=1.0), ffn_norm=_normal(g, (d,), 0.1, mean=1.0))


def _ends(case, seed):
    d, _, _, _, V, _ = DIMS[case["dims"]]
    g = _gen(seed, 1)
    return dict(embed=_normal(g, (V, d), 0.02), lm_head=_normal(g, (V, d), 0.02),
                final_norm=_normal(g, (d,), 0.1, mean=1.0))


def _lengths(b, ctx, seed):
    """The sequences' own lengths: the first has ctx slots, the others up to an eighth fewer."""
    return [ctx - (s * 37 + seed) % max(1, ctx // 8) if s else ctx for s in range(b)]


def _kv_rows(case, seed, layer, seq, n):
    _, H, hd, _, _, _ = DIMS[case["dims"]]
    g = _gen(seed, 1000 + 64 * layer + seq)
    return _normal(g, (H, n, hd), 1.0), _normal(g, (H, n, hd), 1.0)


def _parents(q, width):
    """`width` chains below the root."""
    k = (q - 1) // width
    return [-1] + [0 if i == 0 else w * k + i for w in range(width) for i in range(k)]


def _block(case, seed):
    """The previous block's outputs, from which the next block is built: its newest token and drafts."""
    V = DIMS[case["dims"]][4]
    return _ids(_gen(seed, 2), case.get("b", 1) * case["q"], V - 16)


class _Memory:
    """Device memory of the library as a torch tensor, which keeps its owner alive."""

    def __init__(self, owner, address, shape):
        self.owner = owner
        self.__cuda_array_interface__ = dict(data=(address, False), shape=shape, typestr="<i2", version=2)


def _caches(case, kv):
    _, H, hd, _, _, _ = DIMS[case["dims"]]
    k, v, _, batch, cap = kv.info()
    shape = (case["layers"], batch, H, cap, hd)
    return [torch.as_tensor(_Memory(kv, a, shape), device="cuda").view(torch.bfloat16) for a in (k, v)]


def _model(case, seed, b, cap):
    d, H, hd, F, V, adaptive = DIMS[case["dims"]]
    shape = SimpleNamespace(n_layers=case["layers"], d_model=d, n_heads=H, head_dim=hd, ffn_dim=F, vocab=V,
                            adaptive_id=adaptive, rms_eps=EPS, rope_theta=THETA)
    weights = dict(_ends(case, seed), layers=[_layer(case, seed, l) for l in range(case["layers"])])
    ctx = sd.Context(shape, weights, max_position=cap)
    return ctx, ctx.kv(b, cap)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "tree"):
        b, q, V = case["b"], case["q"], DIMS[case["dims"]][4]
        ctx, kv = _model(case, seed, b, case["ctx"] + q + 16)
        lens = _lengths(b, case["ctx"], seed)
        for l in range(case["layers"]):
            for s, n in enumerate(lens):
                ctx.kv_write(kv, l, s, 0, *_kv_rows(case, seed, l, s, n))
        ctx.kv_commit(kv, torch.tensor(lens, dtype=torch.int32, device="cuda"), b)
        rows = [[c[:, s, :, n:n + q] for c in _caches(case, kv)] for s, n in enumerate(lens)]
        st = dict(ctx=ctx, kv=kv, b=b, q=q, rows=rows, prev=_block(case, seed),
                  prev_acc=torch.ones(b, dtype=torch.int32, device="cuda"),
                  tokens=torch.empty(b * q, dtype=torch.int32, device="cuda"),
                  logits=torch.empty(b * q, V, device="cuda"))
        if kind == "tree":
            st["parent"] = torch.tensor(_parents(q, case["width"]) * b, dtype=torch.int32, device="cuda")
        elif case["accept"]:
            st.update(acc=torch.empty(b, dtype=torch.int32, device="cuda"), out=torch.empty_like(st["tokens"]))
        return st
    if kind == "prompt":
        n, q, V = case["n"], case["q"], DIMS[case["dims"]][4]
        ctx, kv = _model(case, seed, 1, n + q + 16)
        rows = [c[:, 0, :, :n + q] for c in _caches(case, kv)]
        return dict(ctx=ctx, kv=kv, q=q, rows=rows, prompt=_ids(_gen(seed, 3), n, V - 16), block=_block(case, seed),
                    zero=torch.zeros(1, dtype=torch.int32, device="cuda"), logits=torch.empty(q, V, device="cuda"))
    if kind == "attn":
        b, q, H, hd, g = case["b"], case["q"], case["heads"], case["hd"], _gen(seed)
        cap = case["ctx"] + q
        shape = SimpleNamespace(n_layers=1, d_model=H * hd, n_heads=H, head_dim=hd, ffn_dim=256, vocab=256,
                                adaptive_id=0, rms_eps=EPS, rope_theta=THETA)
        return dict(ctx=sd.Context(shape, None, max_position=64), dims=(b, q, H, hd, cap),
                    x=_normal(g, (b * q, H * hd), 1.0, torch.float32), k=_normal(g, (b, H, cap, hd), 1.0),
                    v=_normal(g, (b, H, cap, hd), 1.0), out=torch.empty(b * q, H * hd, device="cuda"),
                    lens=torch.tensor(_lengths(b, case["ctx"], seed), dtype=torch.int32, device="cuda"))
    if kind == "gemm":
        g, shape = _gen(seed), SimpleNamespace(n_layers=1, d_model=128, n_heads=1, head_dim=128, ffn_dim=256,
                                               vocab=256, adaptive_id=0, rms_eps=EPS, rope_theta=THETA)
        return dict(ctx=sd.Context(shape, None, max_position=64), x=_normal(g, (case["M"], case["K"]), 1.0, torch.float32),
                    w=_normal(g, (case["N"], case["K"]), 0.02), y=torch.empty(case["M"], case["N"], device="cuda"))
    b, q, V, g = case["b"], case["q"], case["vocab"], _gen(seed)
    shape = SimpleNamespace(n_layers=1, d_model=128, n_heads=1, head_dim=128, ffn_dim=256, vocab=V, adaptive_id=0,
                            rms_eps=EPS, rope_theta=THETA)
    ctx = sd.Context(shape, None, max_position=4096)
    kv = ctx.kv(b, 2048)
    ctx.kv_commit(kv, torch.tensor(_lengths(b, 1024, seed), dtype=torch.int32, device="cuda"), b)
    logits = _normal(g, (b * q, V), 1.3, torch.float32)
    # drafts as a trained model makes them: seven of ten are the row before's best token
    best = torch.roll(logits.argmax(1).to(torch.int32), 1)
    drafts = torch.where(torch.rand(b * q, generator=g, device="cuda") < 0.7, best, _ids(g, b * q, V))
    return dict(ctx=ctx, kv=kv, logits=logits, drafts=drafts, seed=seed, acc=torch.empty(b, dtype=torch.int32, device="cuda"),
                out=torch.empty(b * q, dtype=torch.int32, device="cuda"), case=case)


def run(s):
    ctx = s["ctx"]
    if "parent" in s:      # a tree block
        ctx.block_forward_tree(s["kv"], s["prev"], s["parent"], s["logits"], s["b"], s["q"])
        return s["logits"], s["rows"]
    if "prev" in s:        # a chain block
        ctx.build_block(s["kv"], 2, s["prev"], s["prev_acc"], s["tokens"], s["b"], s["q"])
        ctx.block_forward(s["kv"], s["tokens"], s["logits"], s["b"], s["q"])
        if "out" not in s:
            return s["logits"], s["rows"]
        ctx.accept_greedy(s["kv"], s["logits"], s["tokens"], s["b"], s["q"], s["q"] - 1, s["acc"], s["out"], commit=False)
        return s["logits"], s["rows"], s["acc"], s["out"]
    if "prompt" in s:      # a prompt, from an empty cache, then the first block
        ctx.kv_commit(s["kv"], s["zero"], 1)
        ctx.prefill(s["kv"], 0, s["prompt"])
        ctx.block_forward(s["kv"], s["block"], s["logits"], 1, s["q"])
        return s["logits"], s["rows"]
    if "lens" in s:
        b, q, H, hd, cap = s["dims"]
        ctx.op_attention(s["x"], s["k"], s["v"], s["lens"], b, q, H, hd, cap, s["out"])
        return s["out"]
    if "w" in s:
        ctx.op_gemm(s["x"], s["w"], s["y"])
        return s["y"]
    c = s["case"]
    if c["temperature"] > 0:
        ctx.accept_nucleus(s["kv"], s["logits"], s["drafts"], c["b"], c["q"], c["q"] - 1, c["top_p"], c["temperature"],
                           s["seed"], s["acc"], s["out"], top_k=c["top_k"], commit=False)
    else:
        ctx.accept_greedy(s["kv"], s["logits"], s["drafts"], c["b"], c["q"], c["q"] - 1, s["acc"], s["out"], commit=False)
    return s["acc"], s["out"]


# ---- what a pass cannot do without, and how close it has to come -----------------------------------


def work(case):
    kind = case["kind"]
    if kind in ("step", "tree", "prompt"):
        d, H, hd, F, V, _ = DIMS[case["dims"]]
        R, L, q = H * hd, case["layers"], case["q"]
        per_layer = 4 * R * d + 3 * d * F
        b = case.get("b", 1)
        lens = _lengths(b, case["ctx"], 0) if "ctx" in case else [case["n"]]
        n = case.get("n", 0)
        rows = b * q
        read = 0 if n else sum(lens)     # a prompt's own rows are written here, not read from before
        bytes_ = 2 * L * per_layer + 2 * V * d + 2 * (rows + n) * d + 4 * L * R * (read + rows + n) + 4 * rows * V
        pairs = sum(q * m + q * (q + 1) // 2 for m in lens) + n * (n + 1) // 2
        flops = 2 * L * per_layer * (rows + n) + 2 * V * d * rows + 4 * L * R * pairs
        return dict(bytes=bytes_, flops=flops)
    if kind == "attn":
        lens, q, R = _lengths(case["b"], case["ctx"], 0), case["q"], case["heads"] * case["hd"]
        return dict(bytes=sum(4 * R * (m + q) + 8 * q * R for m in lens),
                    flops=sum(4 * R * (q * m + q * (q + 1) // 2) for m in lens))
    if kind == "gemm":
        M, K, N = case["M"], case["K"], case["N"]
        return dict(bytes=2 * N * K + 4 * M * (K + N), flops=2 * M * N * K)
    rows = case["b"] * case["q"]
    return dict(bytes=4 * rows * case["vocab"], flops=2 * rows * case["vocab"])


def tolerance(case):
    kind = case["kind"]
    if kind == "accept":
        return "exact"      # the sampler is defined bit for bit
    if kind in ("step", "tree", "prompt"):
        # fp32 sums and bf16 hi + lo operands, but the cache holds bf16 rows: a sum in another
        # order moves some of them by one place.  Measured against 64 bits: 2.4e-3 for block
        # steps and 5.7e-3 for prompts, whose rows all go through the cache.
        return dict(rel=4e-3, max=0.1) if kind != "prompt" else dict(rel=1e-2, max=0.25)
    return dict(rel=2e-5, max=4e-4)     # fp32 sums, operands as bf16 hi + lo (16 bits): 3e-6 to 5e-6 off


# ---- 64 bits ----------------------------------------------------------------------------------------


def _norm(h, gain):
    return h * torch.rsqrt((h * h).mean(-1, keepdim=True) + EPS) * gain


def _rope(x, pos, hd):
    """x [rows, H, hd], rotate-half pairing."""
    inv = THETA ** (-torch.arange(0, hd, 2, dtype=torch.float64, device="cuda") / hd)
    ang = pos.double()[:, None] * inv[None]
    c, s = ang.cos()[:, None], ang.sin()[:, None]
    a, b = x[..., :hd // 2], x[..., hd // 2:]
    return torch.cat([a * c - b * s, b * c + a * s], -1)


def _attend(q, k, v, visible):
    """q [rows, H, hd], k and v [H, keys, hd], visible [rows, keys]."""
    s = torch.einsum("rhd,hkd->hrk", q, k) / math.sqrt(q.shape[-1])
    s = s.masked_fill_(~visible[None], -math.inf).softmax(-1)
    return torch.einsum("hrk,hkd->rhd", s, v)


def _decoder(case, seed, seqs):
    """seqs: per sequence (tokens, positions, cached rows, visible [rows, cached + rows])."""
    d, H, hd, _, _, _ = DIMS[case["dims"]]
    ends = _ends(case, seed)
    toks = torch.cat([t for t, _, _, _ in seqs]).long()
    pos = torch.cat([p for _, p, _, _ in seqs])
    h = ends["embed"][toks].double()
    cut = [len(t) for t, _, _, _ in seqs]
    new = [[[], []] for _ in seqs]
    for l in range(case["layers"]):
        w = _layer(case, seed, l)
        lin = lambda x, n: x @ w[n].double().t()  # noqa: E731
        x = _norm(h, w["attn_norm"].double())
        qh = _rope(lin(x, "wq").view(-1, H, hd), pos, hd)
        kh = _rope(lin(x, "wk").view(-1, H, hd), pos, hd)
        vh = lin(x, "wv").view(-1, H, hd)
        o = []
        for s, (q, k, v) in enumerate(zip(qh.split(cut), kh.split(cut), vh.split(cut))):
            k, v, cached = k.transpose(0, 1), v.transpose(0, 1), seqs[s][2]
            new[s][0].append(k)
            new[s][1].append(v)
            if cached:
                ck, cv = _kv_rows(case, seed, l, s, cached)
                k, v = torch.cat([ck.double(), k], 1), torch.cat([cv.double(), v], 1)
            o.append(_attend(q, k, v, seqs[s][3]))
        h = h + lin(torch.cat(o).reshape(-1, H * hd), "wo")
        x = _norm(h, w["ffn_norm"].double())
        h = h + lin(torch.nn.functional.silu(lin(x, "w_gate")) * lin(x, "w_up"), "w_down")
        del w
    x = _norm(h, ends["final_norm"].double())
    rows = [[torch.stack(c) for c in kv] for kv in new]
    return x, ends["lm_head"].double(), rows


def _seen(cached, rows, parents=None):
    """Which of the cached slots and block rows each block row attends."""
    if parents is None:
        own = torch.ones(rows, rows, dtype=torch.bool, device="cuda").tril()
    else:
        own = torch.zeros(rows, rows, dtype=torch.bool)
        for j in range(rows):
            i = j
            while i >= 0:
                own[j, i] = True
                i = parents[i]
        own = own.cuda()
    return torch.cat([torch.ones(rows, cached, dtype=torch.bool, device="cuda"), own], 1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "tree"):
        q, b = case["q"], case["b"]
        parents = _parents(q, case["width"]) if kind == "tree" else None
        depth = torch.zeros(q, dtype=torch.int64, device="cuda")
        for j in range(1, q):
            depth[j] = depth[parents[j]] + 1 if parents else j
        toks = _block(case, seed).view(b, q)
        seqs = [(toks[s], n + depth, n, _seen(n, q, parents)) for s, n in enumerate(_lengths(b, case["ctx"], seed))]
        x, head, rows = _decoder(case, seed, seqs)
        return (x @ head.t(), rows) + ((None, None) if case.get("accept") else ())
    if kind == "prompt":
        n, q = case["n"], case["q"]
        toks = torch.cat([_ids(_gen(seed, 3), n, DIMS[case["dims"]][4] - 16), _block(case, seed)])
        x, head, rows = _decoder(case, seed, [(toks, torch.arange(n + q, device="cuda"), 0, _seen(0, n + q))])
        return x[n:] @ head.t(), rows[0]
    if kind == "attn":
        b, q, H, hd, g = case["b"], case["q"], case["heads"], case["hd"], _gen(seed)
        cap = case["ctx"] + q
        x = _normal(g, (b * q, H * hd), 1.0, torch.float32).double().view(b, q, H, hd)
        k, v = _normal(g, (b, H, cap, hd), 1.0), _normal(g, (b, H, cap, hd), 1.0)
        out = [_attend(x[s], k[s, :, :n + q].double(), v[s, :, :n + q].double(), _seen(n, q))
               for s, n in enumerate(_lengths(b, case["ctx"], seed))]
        return torch.cat(out).reshape(b * q, H * hd)
    if kind == "gemm":
        g = _gen(seed)
        x = _normal(g, (case["M"], case["K"]), 1.0, torch.float32)
        return x.double() @ _normal(g, (case["N"], case["K"]), 0.02).double().t()
    return None
