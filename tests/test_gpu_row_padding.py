"""Block forwards whose row count lies at the edges of the decode GEMM's operand padding (8, 16,
24, 32 and 64 rows): every sequence of a batch against the same sequence alone, logits and
the K / V rows written."""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2403_18647_gb300 as sd
    shape = synth.SHAPES["tiny"]
    return sd.Context(shape, synth.make_model(shape, seed=0, device="cuda", gain_std=0.1), max_position=256)


def _filled(ctx, b, lens, seqs):
    shape, kv = ctx.shape, ctx.kv(b, 200)
    for i, s in enumerate(seqs):
        for l in range(shape.n_layers):
            k, v = (synth.kv_values(100 + s, l, w, (shape.n_heads, lens[s], shape.head_dim), device="cuda") for w in (0, 1))
            ctx.kv_write(kv, l, i, 0, k, v)
    ctx.kv_commit(kv, torch.tensor([lens[s] for s in seqs], dtype=torch.int32, device="cuda"), b)
    return kv


@pytest.mark.parametrize("b,q", [(1, 7), (1, 8), (1, 9), (2, 8), (1, 16), (3, 8), (5, 5), (2, 16), (3, 11), (3, 16),
                                 (7, 7), (4, 16)])
def test_batch_equals_single_sequences(ctx, b, q):
    shape, lens = ctx.shape, [60 + 17 * s for s in range(b)]
    toks = synth.uniform_ids(3, b * 16 + q, b * q, shape.vocab, device="cuda")
    kv, lg = _filled(ctx, b, lens, range(b)), torch.full((b * q, shape.vocab), float("nan"), device="cuda")
    ctx.block_forward(kv, toks, lg, b, q)
    for s in range(b):
        one, l1 = _filled(ctx, 1, lens, [s]), torch.empty(q, shape.vocab, device="cuda")
        ctx.block_forward(one, toks[s * q:(s + 1) * q].contiguous(), l1, 1, q)
        got = lg[s * q:(s + 1) * q]
        # the same operands in fp32 sums of another order; a cached row's bf16 rounding may flip
        assert ((got - l1).norm() / l1.norm()).item() <= 2e-3
        for l in range(shape.n_layers):
            for x, y in zip(ctx.kv_read(kv, l, s, lens[s], q), ctx.kv_read(one, l, 0, lens[s], q)):
                assert (x.float() - y.float()).abs().max().item() <= 1e-2 * y.float().abs().max().item()
    assert ctx.get_error() == 0


@pytest.mark.parametrize("M", [1, 8, 9, 16, 17, 24, 25, 32, 33, 48, 49, 64])
def test_gemm_row_padding(ctx, M):
    K, N = 4096, 1500   # split tiles, ragged N
    x, w = synth.normal_f32(12, M, (M, K), 1.0, device="cuda"), synth.normal_bf16(12, 1, (N, K), 0.02, device="cuda")
    y = torch.full((M, N), float("nan"), device="cuda")
    ctx.op_gemm(x, w, y)
    ref = x.double() @ w.double().t()
    tol = 5e-5 * K ** 0.5 * 0.02 + 1e-6 * ref.abs().max().item()   # as the other GEMM parity tests
    assert (y.double() - ref).abs().max().item() <= tol
