"""The merge of a step's splits in all its forms (few parts, many, few rows in many parts), on partials made up here: against
the fp64 merge of the same numbers, empty parts among them."""
import pytest
import torch

from paper_2512_10310_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def handle():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    h = B.evlnCreate(0)
    yield h
    B.evlnDestroy(h)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("hq,hkv,d,n,splits", [
    (28, 4, 128, 73, 4),           # the most parts of the first form
    (28, 4, 128, 73, 5),           # one more
    (28, 4, 128, 74, 9),
    (28, 4, 128, 86, 4),           # 4 parts of 602 blocks: the form with the loop
    (28, 4, 128, 170, 3),          # ... of 1190 blocks: without it again
    (28, 4, 128, 21, 5),           # 588 rows: a block per row; in fp32 up to 1000, from 9 parts on up to 1280 rows
    (28, 4, 128, 22, 8),
    (28, 4, 128, 45, 9),           # 1260 rows
    (28, 4, 128, 46, 9),           # 1288 rows
    (28, 4, 128, 8, 16),           # all parts on their way at once
    (28, 4, 128, 8, 17),           # ... and one more
    (3, 1, 128, 1, 32),            # one token, the most parts
    (14, 2, 64, 9, 13),            # two warps per row
    (3, 3, 64, 1, 32),             # an odd number of rows
    (28, 4, 64, 300, 7),
])
def test_merge_against_fp64(handle, dtype, hq, hkv, d, n, splits):
    gen = torch.Generator(device=DEV).manual_seed(1000 * splits + n)
    p = B.step_params(dtype, hq, hkv, d, 32 * 64, n, 32 * 64 + n, 1e4, num_splits=splits)
    assert B.evlnStepNumSplits(handle, p) == splits
    rows = n * hq // hkv
    o = torch.randn((splits, hkv, rows, d), generator=gen, device=DEV)
    lse = 3.0 * torch.randn((splits, hkv, rows), generator=gen, device=DEV)
    empty = torch.rand((splits, hkv, rows), generator=gen, device=DEV) < 0.2
    empty[0] = False                                       # (no row is without keys)
    lse[empty] = float("-inf")
    o[empty] = 0.0
    ws = torch.cat([o.flatten(), lse.flatten()])
    ws = torch.cat([ws, torch.zeros(max(0, (B.evlnStepWorkspaceSize(handle, p) - ws.numel() * 4 + 3) // 4), device=DEV)])
    out = torch.empty((n, hq, d), dtype=torch.bfloat16 if dtype == "bf16" else torch.float32, device=DEV)
    got_lse = torch.empty((n, hq), device=DEV)
    B.evlnStepCombine(handle, p, ws, out, got_lse)
    total = torch.logsumexp(lse.double(), 0)
    want = (torch.exp(lse.double() - total).unsqueeze(-1) * o.double()).sum(0)
    to_tokens = lambda t: t.reshape(hkv, n, hq // hkv, -1).permute(1, 0, 2, 3).reshape(n, hq, -1)
    want, total = to_tokens(want), to_tokens(total)[..., 0]
    # a weight is within some units of 2^-24, a sum of at most 32 products of them within 32 more; then one rounding
    eps = 2.0 ** -8 if dtype == "bf16" else 0.0
    assert bool(((out.double() - want).abs() <= eps * want.abs() + 40 * 2.0 ** -24 * 4.0).all())
    assert float((got_lse.double() - total).abs().max()) <= 16 * 2.0 ** -24 * float(total.abs().max().clamp(min=1.0))


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("hq,hkv,d,n,splits", [
    (28, 4, 128, 45, 12),          # 1260 rows: a block per row
    (28, 4, 128, 74, 12),          # 2072 rows: a warp per row
    (14, 2, 64, 9, 17),
])
def test_parts_of_no_weight_are_left_out(handle, dtype, hq, hkv, d, n, splits):
    # a part from the fifth on whose weight underflows to 0 holds infinite and undefined values: not in the sum, whatever the form
    gen = torch.Generator(device=DEV).manual_seed(7 * splits + n)
    p = B.step_params(dtype, hq, hkv, d, 32 * 64, n, 32 * 64 + n, 1e4, num_splits=splits)
    rows = n * hq // hkv
    o = torch.randn((splits, hkv, rows, d), generator=gen, device=DEV)
    lse = 3.0 * torch.randn((splits, hkv, rows), generator=gen, device=DEV)
    none = torch.rand((splits, hkv, rows), generator=gen, device=DEV) < 0.3
    none[:4] = False
    none[4] = True
    lse[none] = -200.0
    o[none] = 0.0
    outs = []
    for filler in (0.0, float("inf"), float("nan")):
        part = o.clone()
        part[none] = filler
        ws = torch.cat([part.flatten(), lse.flatten()])
        ws = torch.cat([ws, torch.zeros(max(0, (B.evlnStepWorkspaceSize(handle, p) - ws.numel() * 4 + 3) // 4), device=DEV)])
        out = torch.empty((n, hq, d), dtype=torch.bfloat16 if dtype == "bf16" else torch.float32, device=DEV)
        B.evlnStepCombine(handle, p, ws, out, None)
        outs.append(out)
    assert bool(torch.isfinite(outs[0]).all())
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
