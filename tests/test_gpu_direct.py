"""Steps whose keys are not split: the one-call form writes the output from the attention kernel, the three
calls go through the workspace, whose partials are part of the contract.  Same bits, and both against the oracle; sizes at the edges of the
256-row units (several of them start largest first)."""
import dataclasses

import pytest
import torch

from paper_2512_10310_b200 import binding as B
from paper_2512_10310_b200 import workloads as W
from tests.helpers import GpuStep, check_cache, check_output, oracle_step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handle():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    h = B.evlnCreate(0)
    yield h
    B.evlnDestroy(h)


@pytest.mark.parametrize("L,n,splits", [
    (0, 256, 1),        # instruction prefill: 7 units per kv head
    (0, 19, 1),         # 133 rows: just past one tile, a single unit
    (130, 37, 1),       # 259 rows: the second unit has three
    (500, 1100, 0),     # 31 units per kv head: more work items than SM pairs, the library does not split
])
def test_unsplit_step_writes_the_output_directly(handle, L, n, splits):
    cfg = dataclasses.replace(W.STEP_7B, name=f"direct_{L}_{n}", cache_len=L, num_new=n, seed=800 + L + n)
    x = W.make_step_inputs(cfg)
    r = oracle_step("bf16", x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], L, cfg.rope_theta)
    bits = []
    for fused in (True, False):
        gs = GpuStep(handle, "bf16", 28, 4, 128, L + n + 3, cfg.rope_theta, n, num_splits=splits, fused=fused)
        gs.load_cache(x["k_cache"], x["v_cache"])
        g = gs.step(L, x["q_new"], x["k_new"], x["v_new"])
        assert g["splits"] == 1
        check_cache(gs, r, L, n)
        check_output("bf16", g["out"], g["lse"], r["out"], r["lse"])
        bits.append((g["out"].view(torch.int16), g["lse"]))
    assert all(torch.equal(a, b) for a, b in zip(*bits))


@pytest.mark.parametrize("L,n,splits", [
    (1000, 256, 3),     # 84 work items of three or four tiles: persistent pairs that keep their place among the splits
    (0, 256, 3),        # 84 items again, but the units have one or two tiles: empty splits
    (0, 400, 32),       # nearly all of them empty
    (130, 700, 2),      # the first unit has just as many tiles as there are splits
])
def test_more_split_items_than_pairs(handle, L, n, splits):
    cfg = dataclasses.replace(W.STEP_7B, name=f"split_items_{L}_{n}", cache_len=L, num_new=n, seed=900 + L + n)
    x = W.make_step_inputs(cfg)
    r = oracle_step("bf16", x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], L, cfg.rope_theta)
    for fused in (True, False):
        gs = GpuStep(handle, "bf16", 28, 4, 128, L + n + 3, cfg.rope_theta, n, num_splits=splits, fused=fused)
        gs.load_cache(x["k_cache"], x["v_cache"])
        g = gs.step(L, x["q_new"], x["k_new"], x["v_new"])         # (checks the device status)
        assert g["splits"] == splits
        check_cache(gs, r, L, n)
        check_output("bf16", g["out"], g["lse"], r["out"], r["lse"])


@pytest.mark.parametrize("dtype,hq,hkv,d,L,n,splits", [
    ("bf16", 28, 4, 128, 0, 256, 1),       # unsplit on CTA pairs
    ("bf16", 28, 4, 128, 500, 1100, 1),    # ... on persistent ones
    ("bf16", 28, 4, 128, 1000, 196, 3),
    ("bf16", 28, 4, 128, 900, 10, 4),      # the one-CTA kernel
    ("bf16", 28, 4, 128, 900, 1, 1),       # few rows
    ("f32", 4, 2, 64, 300, 40, 2),
])
def test_workspace_holds_the_partials(handle, dtype, hq, hkv, d, L, n, splits):
    # what evlnStepAttention leaves is documented: [S, Hkv, n G, D] outputs, then [S, Hkv, n G] log-sum-exps, all
    # float.  A caller's own merge of them is what evlnStepCombine gives, up to its fp32 sums and one rounding.
    cfg = W.StepConfig("partials", dtype, hq, hkv, d, L, n, 1e6, 0.5, 60 + L + n)
    x = W.make_step_inputs(cfg)
    gs = GpuStep(handle, dtype, hq, hkv, d, L + n, cfg.rope_theta, n, num_splits=splits)
    gs.load_cache(x["k_cache"], x["v_cache"])
    g = gs.step(L, x["q_new"], x["k_new"], x["v_new"])
    p, rows = gs.params(L, n), n * hq // hkv
    q_rot = g["q_rot"].reshape(n, hkv, hq // hkv, d).permute(1, 0, 2, 3).contiguous()
    ws = torch.full((B.evlnStepWorkspaceSize(handle, p) // 4,), float("nan"), device="cuda:0")
    B.evlnStepAttention(handle, p, q_rot, gs.k_cache, gs.v_cache, ws)
    o = ws[:splits * hkv * rows * d].view(splits, hkv, rows, d).double()
    lse = ws[splits * hkv * rows * d:][:splits * hkv * rows].view(splits, hkv, rows).double()
    total = torch.logsumexp(lse, 0)
    out = (torch.exp(lse - total).unsqueeze(-1) * o).sum(0)
    to_tokens = lambda t: t.reshape(hkv, n, hq // hkv, -1).permute(1, 0, 2, 3).reshape(n, hq, -1)
    eps = 2.0 ** -8 if dtype == "bf16" else 1e-6           # half a unit of the storage type, and the sums' last bits
    assert bool(((g["out"].double() - to_tokens(out)).abs() <= eps * to_tokens(out).abs() + 1e-6).all())
    assert float((g["lse"].double() - to_tokens(total)[..., 0]).abs().max()) <= 1e-5


@pytest.mark.parametrize("hq,hkv,L,n,unsplit", [
    (28, 4, 128, 196, True),      # three key tiles, many rows: the merge costs more than it saves
    (28, 4, 0, 40, True),         # one tile
    (28, 4, 700, 40, False),      # six tiles, few rows: unsplit, three calls took 12.5 us against 10.6
    (32, 8, 700, 64, False),
])
def test_where_short_steps_are_split(handle, hq, hkv, L, n, unsplit):
    p = B.step_params("bf16", hq, hkv, 128, L, n, L + n, 1e6)
    assert (B.evlnStepNumSplits(handle, p) == 1) == unsplit
