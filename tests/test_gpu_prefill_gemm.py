"""The prefill GEMM (CTA pairs, tiles split along K) at the sizes where its work list changes
shape: one tile, an odd number of weight tiles, fewer tiles than pairs, a split remainder
before whole tiles, whole tiles only, ragged K, N and positions.  Reference: fp64 product."""
import math

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2403_18647_gb300 as sd
    shape = synth.SHAPES["tiny"]
    return sd.Context(shape, synth.make_model(shape, seed=0, device="cuda"), max_position=64)


@pytest.mark.parametrize("M,K,N", [
    (65, 8, 1), (65, 512, 128), (100, 4096, 4096), (128, 704, 384), (129, 4096, 640), (512, 72, 20000),
    (500, 2056, 12288), (97, 11008, 4096), (511, 4096, 9856), (160, 5120, 15361), (512, 1024, 38912)])
def test_prefill_gemm_work_lists(ctx, M, K, N):
    x = synth.normal_f32(3, M, (M, K), 1.0, device="cuda")
    w = synth.normal_bf16(3, 7 + N, (N, K), 0.02, device="cuda")
    y = torch.full((M, N), float("nan"), device="cuda")
    again = torch.full_like(y, float("nan"))
    ctx.op_gemm(x, w, y)
    ctx.op_gemm(x, w, again)   # the tile counters are back at zero
    assert ctx.get_error() == 0
    assert torch.equal(y, again)
    ref = x.double() @ w.double().t()
    # the operand's hi + lo split (2^-16 relative) and the fp32 accumulation, as for the other GEMMs
    tol = 5e-5 * math.sqrt(K) * 0.02 + 1e-6 * ref.abs().max().item()
    err = (y.double() - ref).abs().max().item()
    assert err <= tol, (err, tol)
