"""Steps whose keys are not split: the one-call form writes the output from the attention kernel, the three
calls go through the workspace.  Same bits, and both against the oracle; sizes at the edges of the
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
