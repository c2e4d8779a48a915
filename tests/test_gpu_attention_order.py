"""sdsat_op_attention right behind kernels that let their dependents start before they write: a
commit, a prefill, a tree commit with its compaction, and the caller's own copies.  The attention
reads the lengths and rows that those leave; nothing synchronises in between."""
import math

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


class _Memory:
    def __init__(self, address, shape, typestr):
        self.__cuda_array_interface__ = dict(data=(address, False), shape=shape, typestr=typestr, version=2)


def _views(kv, shape):
    """The last layer's caches [b][H][cap][hd] and the committed lengths, in place."""
    k, v, ln, b, cap = kv.info()
    size = shape.n_layers, b, shape.n_heads, cap, shape.head_dim
    caches = [torch.as_tensor(_Memory(a, size, "<i2"), device="cuda").view(torch.bfloat16)[-1] for a in (k, v)]
    return caches + [torch.as_tensor(_Memory(ln, (b,), "<i4"), device="cuda")]


def _softmax(x, k, v, n, q):
    H, hd = k.shape[0], k.shape[2]
    s = torch.einsum("qhd,hkd->hqk", x.double().view(q, H, hd), k[:, :n + q].double()) / math.sqrt(hd)
    seen = torch.ones(q, n + q, dtype=torch.bool, device="cuda").tril(n)
    return torch.einsum("hqk,hkd->qhd", s.masked_fill(~seen, float("-inf")).softmax(-1), v[:, :n + q].double()).reshape(q, H * hd)


@pytest.fixture(scope="module")
def ctx():
    import paper_2403_18647_gb300 as sd
    shape = synth.ModelShape("order", 2, 512, 4, 128, 384, 1000, 999)
    return sd.Context(shape, synth.make_model(shape, seed=1, device="cuda"), max_position=4096)


def _filled(ctx, b, cap):
    shape, kv = ctx.shape, ctx.kv(b, cap)
    for l in range(shape.n_layers):
        for s in range(b):
            ctx.kv_write(kv, l, s, 0, *(synth.kv_values(7 + s, l, w, (shape.n_heads, cap, shape.head_dim), device="cuda") for w in (0, 1)))
    return kv


def _attend(ctx, views, x, b, q):
    k, v, ln = views
    out = torch.full_like(x, float("nan"))
    ctx.op_attention(x, k, v, ln, b, q, ctx.shape.n_heads, ctx.shape.head_dim, k.shape[2], out)
    return out


@pytest.mark.parametrize("q", [6, 11])
def test_attention_behind_a_commit(ctx, q):
    b, cap = 2, 2100
    kv = _filled(ctx, b, cap)
    views = _views(kv, ctx.shape)
    x = synth.normal_f32(5, q, (b * q, 512), 1.0, device="cuda")
    lens = [[16 * i % (cap - q), cap - q - 23 * i] for i in range(1, 40)]
    new = torch.tensor(lens, dtype=torch.int32, device="cuda")
    outs = []
    for i in range(len(lens)):
        ctx.kv_commit(kv, new[i], b)
        outs.append(_attend(ctx, views, x, b, q))
    for o, n in zip(outs, lens):
        for s in range(b):
            ref = _softmax(x[s * q:(s + 1) * q], views[0][s], views[1][s], n[s], q)
            assert (o[s * q:(s + 1) * q].double() - ref).abs().max().item() <= 2e-5   # as the other attention tests
    assert ctx.get_error() == 0


@pytest.mark.parametrize("n", [6, 130])
def test_attention_behind_a_prefill(ctx, n):
    q, cap = 6, 400
    kv = _filled(ctx, 1, cap)
    views = _views(kv, ctx.shape)
    x = synth.normal_f32(6, n, (q, 512), 1.0, device="cuda")
    outs = []
    for i in range(3):
        ctx.prefill(kv, 0, synth.prompt_ids(3, i, n, 900).cuda())
        outs.append(_attend(ctx, views, x, 1, q))
    # slots past a prefill's hold the fill until the next one writes them: the first output is
    # checked against a cache that only the first prefill has touched, and so on
    for i, o in enumerate(outs):
        one = _filled(ctx, 1, cap)
        for j in range(i + 1):
            ctx.prefill(one, 0, synth.prompt_ids(3, j, n, 900).cuda())
        k, v = ctx.kv_read(one, 1, 0, 0, cap)
        assert (o.double() - _softmax(x, k, v, n * (i + 1), q)).abs().max().item() <= 2e-5
    assert ctx.get_error() == 0


def test_attention_behind_a_tree_commit(ctx):
    """The accepted path's rows are moved by the compaction kernel."""
    q, n, cap = 9, 500, 600
    parent = [-1, 0, 0, 1, 2, 3, 4, 5, 6]   # two chains of four; the second one (rows 2, 4, 6, 8) is accepted
    targets = [20, 31, 22, 33, 24, 35, 26, 37, 28]
    tokens = [1, 11, 20, 13, 22, 15, 24, 17, 26]
    lg = torch.zeros(q, ctx.shape.vocab, device="cuda")
    lg[torch.arange(q), torch.tensor(targets)] = 5.0
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")   # noqa: E731
    tok, par, length, x = i32(tokens), i32(parent), i32([n]), synth.normal_f32(7, 1, (6, 512), 1.0, device="cuda")
    acc, out = i32([0]), i32([0] * q)
    for _ in range(10):
        kv = _filled(ctx, 1, cap)
        views = _views(kv, ctx.shape)
        k, v = (c[0].clone() for c in views[:2])
        for c in (k, v):
            c[:, n + 1:n + 5] = c[:, [n + 2, n + 4, n + 6, n + 8]]
        ctx.kv_commit(kv, length, 1)
        ctx.accept_tree(kv, lg, tok, par, 1, q, acc, out)
        o = _attend(ctx, views, x, 1, 6)
        assert (o.double() - _softmax(x, k, v, n + 5, 6)).abs().max().item() <= 2e-5
        assert acc.item() == 5
    assert ctx.get_error() == 0


def test_attention_behind_the_callers_own_kernels(ctx):
    b, q, cap = 1, 6, 2100
    shape = ctx.shape
    x = synth.normal_f32(8, 1, (q, 512), 1.0, device="cuda")
    k, v = (torch.zeros(b, shape.n_heads, cap, shape.head_dim, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    ln = torch.zeros(b, dtype=torch.int32, device="cuda")
    src = [[synth.kv_values(i, 0, w, k.shape, device="cuda") for w in (0, 1)] for i in range(2)]
    outs = []
    for i in range(20):
        k.copy_(src[i % 2][0])
        v.copy_(src[i % 2][1])
        ln.fill_(100 * i)
        outs.append(_attend(ctx, (k, v, ln), x, b, q))
    for i, o in enumerate(outs):
        ref = _softmax(x, src[i % 2][0][0], src[i % 2][1][0], 100 * i, q)
        assert (o.double() - ref).abs().max().item() <= 2e-5
