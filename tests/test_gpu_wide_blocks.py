"""Blocks of 33 to 64 rows against the oracle, on models that differ in which GEMMs of a layer
leave their tiles whole and which end in a second kernel: with the O or down projection whole the
next operand is not normalised yet, and the consuming GEMM (QKV, gate/up, the LM head) applies the
RMSNorm factor of every row.  Then blocks whose attention takes a smaller cluster than fits."""
import numpy as np
import pytest
import torch

import synth
from oracle import model as OM
from oracle import tree as OT

pytestmark = pytest.mark.gpu

# d_model, heads, head_dim, ffn, vocab
SHAPES = {
    "O, down and head whole": (256, 4, 64, 256, 1003),
    "down whole, head with split and whole tiles": (1024, 8, 128, 512, 20500),
    "down whole, head in a second kernel": (1024, 8, 128, 256, 1003),
    "O whole, down in a second kernel": (256, 4, 64, 688, 4104),
}
BLOCKS = [(3, 11), (3, 16), (4, 16)]   # 33, 48 and 64 rows


@pytest.fixture(scope="module", params=list(SHAPES))
def model(request):
    import paper_2403_18647_gb300 as sd
    d, H, hd, F, V = SHAPES[request.param]
    shape = synth.ModelShape("wide", 2, d, H, hd, F, V, V - 1)
    W = OM.Weights(shape, tensors=synth.make_model(shape, seed=0, device="cpu", gain_std=0.1))
    return shape, sd.Context(shape, synth.make_model(shape, seed=0, device="cuda", gain_std=0.1), max_position=256), W


def _compare(model, b, q, lens, cap, parent):
    shape, ctx, W = model
    kv, kvo = ctx.kv(b, cap), OM.KVCache(shape, b, cap, kv_bf16=True)
    for s, n in enumerate(lens):
        for l in range(shape.n_layers):
            rows = [synth.kv_values(100 + s, l, w, (shape.n_heads, n, shape.head_dim), device="cuda") for w in (0, 1)]
            ctx.kv_write(kv, l, s, 0, *rows)
            kvo.K[l][s][:, :n], kvo.V[l][s][:, :n] = (OM.to64(x) for x in rows)
        kvo.len[s] = n
    ctx.kv_commit(kv, torch.tensor(lens, dtype=torch.int32, device="cuda"), b)
    toks = synth.uniform_ids(3, b * 16 + q, b * q, shape.vocab)
    lg = torch.full((b * q, shape.vocab), float("nan"), device="cuda")
    if parent:
        ctx.block_forward_tree(kv, toks.cuda(), torch.tensor(parent * b, dtype=torch.int32, device="cuda"), lg, b, q)
    else:
        ctx.block_forward(kv, toks.cuda(), lg, b, q)
    got = lg.cpu().double().numpy()
    for s in range(b):
        ids = toks[s * q:(s + 1) * q].tolist()
        ref = OT.tree_forward(W, kvo, s, ids, parent) if parent else OM.block_forward(W, kvo, s, ids)
        # per row: a factor of one row must not hide in the others.  Operands as bf16 hi + lo and
        # fp32 sums leave 1e-5; a K or V element whose bf16 rounding falls the other way (2^-8 of
        # it) moves an attention output of some 60 to 130 slots by less than 1e-4
        err = np.linalg.norm(got[s * q:(s + 1) * q] - ref, axis=1) / np.linalg.norm(ref, axis=1)
        assert err.max() <= 2e-3, err
    assert ctx.get_error() == 0


@pytest.mark.parametrize("tree", [False, True], ids=["chain", "tree"])
@pytest.mark.parametrize("b,q", BLOCKS)
def test_wide_block_matches_oracle(model, b, q, tree):
    parent = [-1, 0, 1, 2, 0, 4, 4, 1, 7, 0, 9, 10, 10, 3, 13, 14][:q]
    _compare(model, b, q, [60 + 17 * s for s in range(b)], 200, parent if tree else None)


@pytest.mark.parametrize("q", [6, 14])
def test_block_whose_attention_takes_the_smaller_cluster(q):
    """80 (sequence, head) pairs: clusters of 5 fit, but fewer than a tenth more of them than pairs."""
    import paper_2403_18647_gb300 as sd
    shape = synth.ModelShape("pairs", 1, 512, 40, 128, 384, 1003, 1002)
    W = OM.Weights(shape, tensors=synth.make_model(shape, seed=0, device="cpu", gain_std=0.1))
    ctx = sd.Context(shape, synth.make_model(shape, seed=0, device="cuda", gain_std=0.1), max_position=512)
    _compare((shape, ctx, W), 2, q, [480, 333], 500, None)
