"""Block forwards whose row count lies at the edges of the GEMMs they run on (operand padding to
8, 16, 24 and 32 rows, and from 33 rows the tiled GEMM): every sequence of a batch against the
same sequence alone: logits, the last layer's workspaces and the K / V rows written."""
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


@pytest.mark.parametrize("b,q", [(1, 7), (1, 8), (1, 9), (2, 8), (1, 16), (3, 8), (5, 5), (4, 7), (5, 6), (2, 16), (3, 11), (3, 16),
                                 (7, 7), (4, 16)])
def test_batch_equals_single_sequences(ctx, b, q):
    shape, lens = ctx.shape, [60 + 17 * s for s in range(b)]
    toks = synth.uniform_ids(3, b * 16 + q, b * q, shape.vocab, device="cuda")
    kv, lg = _filled(ctx, b, lens, range(b)), torch.full((b * q, shape.vocab), float("nan"), device="cuda")
    ctx.block_forward(kv, toks, lg, b, q)
    ws = [ctx.debug_workspace(i, b * q) for i in range(4)]
    for s in range(b):
        one, l1 = _filled(ctx, 1, lens, [s]), torch.empty(q, shape.vocab, device="cuda")
        ctx.block_forward(one, toks[s * q:(s + 1) * q].contiguous(), l1, 1, q)
        got = lg[s * q:(s + 1) * q]
        # the same operands in fp32 sums of another order; a cached row's bf16 rounding may flip
        assert ((got - l1).norm() / l1.norm()).item() <= 2e-3
        for i in range(4):
            x, y = ws[i][s * q:(s + 1) * q], ctx.debug_workspace(i, q)
            assert ((x - y).norm() / y.norm()).item() <= 2e-3, i
        for l in range(shape.n_layers):
            for x, y in zip(ctx.kv_read(kv, l, s, lens[s], q), ctx.kv_read(one, l, 0, lens[s], q)):
                assert (x.float() - y.float()).abs().max().item() <= 1e-2 * y.float().abs().max().item()
    assert ctx.get_error() == 0


@pytest.mark.parametrize("b,q", [(2, 11), (3, 11), (4, 15)])
def test_tree_batch_equals_single_sequences(ctx, b, q):
    """Tree blocks: positions and masks follow the parents on either GEMM."""
    shape, lens = ctx.shape, [60 + 17 * s for s in range(b)]
    parent = [-1, 0, 1, 2, 0, 4, 4, 1, 7, 0, 9, 10, 10, 3, 13][:q]
    toks = synth.uniform_ids(4, b * 16 + q, b * q, shape.vocab, device="cuda")
    par = torch.tensor(parent * b, dtype=torch.int32, device="cuda")
    kv, lg = _filled(ctx, b, lens, range(b)), torch.full((b * q, shape.vocab), float("nan"), device="cuda")
    ctx.block_forward_tree(kv, toks, par, lg, b, q)
    for s in range(b):
        one, l1 = _filled(ctx, 1, lens, [s]), torch.empty(q, shape.vocab, device="cuda")
        ctx.block_forward_tree(one, toks[s * q:(s + 1) * q].contiguous(), par[:q].contiguous(), l1, 1, q)
        assert ((lg[s * q:(s + 1) * q] - l1).norm() / l1.norm()).item() <= 2e-3
    assert ctx.get_error() == 0


@pytest.mark.parametrize("M", [25, 32])
@pytest.mark.parametrize("K,N", [(64, 100), (512, 4864), (520, 4864), (512, 4865), (1024, 16897), (1032, 16897), (1024, 38912), (1024, 38913)])
def test_gemm_of_25_to_32_rows(ctx, M, K, N):
    """Skinny and tiled GEMM on both sides of the lines in K and N."""
    x, w = synth.normal_f32(13, M, (M, K), 1.0, device="cuda"), synth.normal_bf16(13, 1, (N, K), 0.02, device="cuda")
    y = torch.full((M, N), float("nan"), device="cuda")
    ctx.op_gemm(x, w, y)
    ref = x.double() @ w.double().t()
    tol = 5e-5 * K ** 0.5 * 0.02 + 1e-6 * ref.abs().max().item()   # as the other GEMM parity tests
    assert (y.double() - ref).abs().max().item() <= tol and ctx.get_error() == 0


def test_wide_block_past_the_capacity(ctx):
    """Rows past the KV capacity on the tiled GEMM: flagged, not written, the others as usual."""
    b, q = 3, 16
    kv = ctx.kv(b, 100)
    ctx.kv_commit(kv, torch.tensor([100 - q, 100 - 5, 0], dtype=torch.int32, device="cuda"), b)
    toks = synth.uniform_ids(5, 1, b * q, ctx.shape.vocab, device="cuda")
    lg = torch.empty(b * q, ctx.shape.vocab, device="cuda")
    ctx.block_forward(kv, toks, lg, b, q)
    assert ctx.get_error() == 0x4
    k, _ = ctx.kv_read(kv, 0, 0, 100 - q, q)
    assert (k.float().abs().sum(dim=(0, 2)) > 0).all()
    k, _ = ctx.kv_read(kv, 0, 1, 0, 100)
    assert (k.float().abs().sum(dim=(0, 2))[:95] == 0).all() and (k.float().abs().sum(dim=(0, 2))[95:] > 0).all()


@pytest.mark.parametrize("M,N", [(M, 1500) for M in (1, 8, 9, 16, 17, 24, 25, 28, 29, 32, 33, 64)] +
                         [(M, N) for M in (25, 32) for N in (4864, 4865, 16896, 16897)])
def test_gemm_row_padding(ctx, M, N):
    K = 4096   # split tiles, ragged N
    x, w = synth.normal_f32(12, M, (M, K), 1.0, device="cuda"), synth.normal_bf16(12, 1, (N, K), 0.02, device="cuda")
    y = torch.full((M, N), float("nan"), device="cuda")
    ctx.op_gemm(x, w, y)
    ref = x.double() @ w.double().t()
    tol = 5e-5 * K ** 0.5 * 0.02 + 1e-6 * ref.abs().max().item()   # as the other GEMM parity tests
    assert (y.double() - ref).abs().max().item() <= tol


@pytest.mark.parametrize("H,hd,ffn", [(9, 128, 1184), (18, 64, 2000)])
def test_second_kernel_of_split_tiles(H, hd, ffn):
    """17 to 24 rows with tiles split along K (d 1152): O, down and QKV end in a second kernel.
    Chains and trees against single sequences, and rows past the capacity."""
    import paper_2403_18647_gb300 as sd
    shape = synth.ModelShape("mid", 2, H * hd, H, hd, ffn, 1003, 1000)
    ctx = sd.Context(shape, synth.make_model(shape, seed=0, device="cuda", gain_std=0.1), max_position=256)
    for b, q in ((6, 3), (4, 5), (7, 3), (4, 6)):
        test_batch_equals_single_sequences(ctx, b, q)
    test_tree_batch_equals_single_sequences(ctx, 2, 11)
    b, q = 2, 10
    kv = ctx.kv(b, 100)
    ctx.kv_commit(kv, torch.tensor([100 - q, 100 - 4], dtype=torch.int32, device="cuda"), b)
    toks = synth.uniform_ids(5, 1, b * q, shape.vocab, device="cuda")
    ctx.block_forward(kv, toks, torch.empty(b * q, shape.vocab, device="cuda"), b, q)
    assert ctx.get_error() == 0x4
    for i, n in ((0, q), (1, 4)):
        for x in ctx.kv_read(kv, 1, i, 0, 100):
            w = x.float().abs().sum(dim=(0, 2))
            assert (w[:100 - n] == 0).all() and (w[100 - n:] > 0).all()
