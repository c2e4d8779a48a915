"""The prefill attention at the edges of its tiles (128 positions, 128 keys) and launch forms
(one or two tiles per CTA, one or two chunks, a cache that already holds slots): the second
layer's K and V rows, which depend on the first layer's attention, against the same prompt fed
as 16-row decode blocks, and against the oracle.  And the sequences of a batch: each prefill
writes its own rows only."""
import dataclasses

import numpy as np
import pytest
import torch

import synth
from oracle import model as OM

pytestmark = pytest.mark.gpu

# heads x head_dim: with 40 heads, more than 768 positions take two tiles per CTA
SHAPES = {(4, 128): 1, (40, 64): 2}


def _model(H, hd):
    import paper_2403_18647_gb300 as sd
    shape = dataclasses.replace(synth.SHAPES["7b"], name="edge", n_layers=2, d_model=512, n_heads=H, head_dim=hd,
                                ffn_dim=384, vocab=1000, adaptive_id=999)
    return shape, sd.Context(shape, synth.make_model(shape, seed=5, device="cuda", gain_std=0.1), max_position=8192)


@pytest.fixture(scope="module", params=list(SHAPES))
def model(request):
    return _model(*request.param)


@pytest.fixture(scope="module")
def wide_model():
    return _model(40, 128)


def _blocks(ctx, kv, ids, start):
    lg = torch.empty(16, 1000, device="cuda")
    for i in range(0, ids.numel(), 16):
        blk = ids[i:i + 16].contiguous()
        ctx.block_forward(kv, blk, lg[:blk.numel()], 1, blk.numel())
        ctx.kv_commit(kv, torch.tensor([start + i + blk.numel()], dtype=torch.int32, device="cuda"), 1)


@pytest.mark.parametrize("start", [0, 37])
@pytest.mark.parametrize("n", [17, 64, 65, 127, 128, 129, 256, 257, 700, 1000, 2200, 4200])
def test_prefill_attention_edges(model, n, start):
    shape, ctx = model
    ids = synth.prompt_ids(7, n, n + start, 900).cuda()
    kvs = [ctx.kv(1, n + start + 8) for _ in range(2)]
    for kv in kvs:
        if start:
            _blocks(ctx, kv, ids[:start].contiguous(), 0)
    ctx.prefill(kvs[0], 0, ids[start:].contiguous())
    _blocks(ctx, kvs[1], ids[start:].contiguous(), start)
    assert ctx.kv_lengths(kvs[0]).item() == n + start and ctx.get_error() == 0
    for a, b in zip(ctx.kv_read(kvs[0], 1, 0, 0, n + start), ctx.kv_read(kvs[1], 1, 0, 0, n + start)):
        a, b = a.float(), b.float()
        # fp32-like sums on both sides; rows differ where a bf16 rounding falls the other way
        # (2^-8 of the value), and through the first layer's such rows
        assert torch.isfinite(a).all()
        assert (a - b).abs().max().item() <= 1e-2 * b.abs().max().item()
        assert ((a - b).norm() / b.norm()).item() <= 2e-3


# two tiles of 128 dimensions per CTA: the last CTA with two tiles, one, and one of a single position
@pytest.mark.parametrize("start", [0, 37])
@pytest.mark.parametrize("n", [1000, 1025, 1100, 2200])
def test_prefill_attention_two_tiles_of_128_dimensions(wide_model, n, start):
    test_prefill_attention_edges(wide_model, n, start)


@pytest.mark.parametrize("lens", [(70, 17, 40), (300, 1100, 129)])
def test_prefill_of_each_sequence(model, lens):
    """Sequences 1, 2 and 0 of one cache: the rows of each are, bit for bit, those of the same prompt
    in a cache of its own, and nothing else in the cache changes."""
    shape, ctx = model
    cap = max(lens) + 9
    kv = ctx.kv(3, cap)
    fill = [[[synth.kv_values(3 + s, l, w, (shape.n_heads, cap, shape.head_dim), device="cuda") for w in (0, 1)]
             for l in range(shape.n_layers)] for s in range(3)]
    for s in range(3):
        for l in range(shape.n_layers):
            ctx.kv_write(kv, l, s, 0, *fill[s][l])
    ids = [synth.prompt_ids(9, s, n, 900).cuda() for s, n in enumerate(lens)]
    for s in (1, 2, 0):
        ctx.prefill(kv, s, ids[s])
    assert ctx.kv_lengths(kv).tolist() == list(lens) and ctx.get_error() == 0
    for s, n in enumerate(lens):
        one = ctx.kv(1, cap)
        ctx.prefill(one, 0, ids[s])
        for l in range(shape.n_layers):
            for got, ref, old in zip(ctx.kv_read(kv, l, s, 0, cap), ctx.kv_read(one, l, 0, 0, cap), fill[s][l]):
                assert torch.equal(got[:, :n], ref[:, :n]) and torch.equal(got[:, n:], old[:, n:])


# one and two tiles of 128 positions per CTA, a last tile of 44 and of 32 positions
@pytest.mark.parametrize("H,hd,n", [(4, 128, 300), (40, 64, 800), (40, 128, 800)])
def test_prefill_attention_matches_oracle(H, hd, n):
    """The second layer's K and V rows, which depend on the first layer's attention."""
    shape, ctx = _model(H, hd)
    W = OM.Weights(shape, tensors=synth.make_model(shape, seed=5, device="cpu", gain_std=0.1))
    ids = synth.prompt_ids(8, n, n, 900)
    kvo = OM.KVCache(shape, 1, n, kv_bf16=True)
    OM.prefill(W, kvo, 0, ids.tolist())
    kv = ctx.kv(1, n + 8)
    ctx.prefill(kv, 0, ids.cuda())
    for got, ref in zip(ctx.kv_read(kv, 1, 0, 0, n), (kvo.K[1][0][:, :n], kvo.V[1][0][:, :n])):
        err = got.float().cpu().double().numpy() - ref
        # both sides store bf16 rows: a rounding that falls the other way is 2^-8 of the value
        assert np.abs(err).max() <= 1e-2 * np.abs(ref).max() and np.linalg.norm(err) <= 2e-3 * np.linalg.norm(ref)
    assert ctx.get_error() == 0
