"""Paged batches at the edges of how their work is dealt out (work items to CTA pairs, equal shares to blocks),
against the oracle."""
import dataclasses

import pytest
import torch

from oracle import step_oracle as so
from paper_2512_10310_b200 import binding as B
from paper_2512_10310_b200 import workloads as W
from tests.helpers import GpuStep, check_output, f64, oracle_step
from tests.test_gpu_paged import _check_pools, _gpu_paged

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handle():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    h = B.evlnCreate(0)
    yield h
    B.evlnDestroy(h)


@pytest.mark.parametrize("batch,heads", [
    (4, 16),       # 64 work items: fewer than SM pairs, a launch without persistent pairs
    (37, 2),       # 74: as many as pairs
    (38, 2),       # 76: more
    (20, 16),      # 320: dealt to the pairs by the item table
    (64, 16),      # 1024: more than the table holds, dealt in turn
    (160, 16),     # 2560: more than the pairs keep, two launches
])
def test_paged_batch_of_many_work_items(handle, batch, heads):
    # one query head per kv head and 33 tokens: one unit per (episode, kv head) for the tile kernel
    cfg = dataclasses.replace(W.PAGED_B16, name=f"many_{batch}", num_q_heads=heads, num_kv_heads=heads, batch=batch, seed=90 + batch)
    lens = [(37 * b) % 301 for b in range(batch)]
    x = W.make_paged_inputs(cfg, lens, [33] * batch)
    out, lse, k_pool, v_pool = _gpu_paged(handle, cfg, x)
    okp, ovp = f64(x["k_pool"]), f64(x["v_pool"])
    ref_out, ref_lse = so.step_paged(f64(x["q_new"]), f64(x["k_new"]), f64(x["v_new"]), okp, ovp, x["page_table"], lens,
                                     x["new_offsets"], cfg.rope_theta, storage="bf16")
    check_output("bf16", out, lse, ref_out, ref_lse)
    _check_pools(x, cfg, k_pool, v_pool, okp, ovp)


@pytest.mark.parametrize("hq,hkv,lens,new", [
    (28, 4, [5], [1]),                                        # shares of one stage
    (28, 4, [64, 0, 700, 63, 4000], [0, 2, 0, 1, 4]),         # shares go over episodes without new tokens; two row tiles
    (7, 1, [32000], [1]),                                     # a row in as many parts as a warp merges
    (64, 8, [900, 2000, 130], [4, 1, 3]),                     # more work items per token than a block has threads
    (4, 4, [(53 * b) % 190 for b in range(200)], [1] * 200),  # shares of many short units
])
def test_paged_batch_of_few_rows_in_equal_shares(handle, hq, hkv, lens, new):
    cfg = dataclasses.replace(W.PAGED_B16, name="shares", num_q_heads=hq, num_kv_heads=hkv, batch=len(lens), seed=120 + len(lens))
    x = W.make_paged_inputs(cfg, lens, new)
    out, lse, k_pool, v_pool = _gpu_paged(handle, cfg, x)
    okp, ovp = f64(x["k_pool"]), f64(x["v_pool"])
    ref_out, ref_lse = so.step_paged(f64(x["q_new"]), f64(x["k_new"]), f64(x["v_new"]), okp, ovp, x["page_table"], lens,
                                     x["new_offsets"], cfg.rope_theta, storage="bf16")
    check_output("bf16", out, lse, ref_out, ref_lse)
    _check_pools(x, cfg, k_pool, v_pool, okp, ovp)


@pytest.mark.parametrize("hq,hkv,length,new,least", [
    (7, 1, 20000, 64, 12),        # two row units of one kv head: in up to 8 parts 26.0 us, in as many as pay 18.7
    (28, 4, 9000, 20, 9),
    (28, 4, 700, 196, 1),
])
def test_paged_frame_of_one_long_episode(handle, hq, hkv, length, new, least):
    cfg = dataclasses.replace(W.PAGED_B16, name="long", num_q_heads=hq, num_kv_heads=hkv, batch=1, seed=140 + new)
    x = W.make_paged_inputs(cfg, [length], [new])
    p = B.paged_params(hq, hkv, 128, 1, 64, x["num_pages"], len(x["page_table"][0]), cfg.rope_theta)
    parts = B.evlnPagedWorkspaceSize(handle, p, [length], [0, new]) // (new * hq * 129 * 4)
    assert parts >= least
    out, lse, k_pool, v_pool = _gpu_paged(handle, cfg, x)
    okp, ovp = f64(x["k_pool"]), f64(x["v_pool"])
    ref_out, ref_lse = so.step_paged(f64(x["q_new"]), f64(x["k_new"]), f64(x["v_new"]), okp, ovp, x["page_table"], [length],
                                     x["new_offsets"], cfg.rope_theta, storage="bf16")
    check_output("bf16", out, lse, ref_out, ref_lse)
    _check_pools(x, cfg, k_pool, v_pool, okp, ovp)


RISING = [(130, 17.0), (200, 34.0), (300, 51.0), (420, 68.0)]      # (token, its key): second tile, both halves, third, fourth


def _rising_scores(q, k, starts, lengths):
    # each of these keys is 60 above the one before for all queries, so a row's reference moves at each of them
    q[:, :, 63], q[:, :, 127] = 40.0, 0.0       # the channel that turns least
    k[:, :, 63] = 0.0
    for start, n in zip(starts, lengths):
        for tok, value in RISING:
            if tok < n:
                k[start + tok, :, 63] = value


def test_references_move_in_later_items_of_a_pair(handle):
    # 232 work items on contiguous caches: a pair's second and third start while rows of the one before are still to be read
    # (0.3: a bf16 operand's rounding grows with the logits that it makes, 1.04 % of a row's rms at 1.0, and values up to 4 are rounded by
    # more than the absolute gate; neither is what is tested)
    cfg = dataclasses.replace(W.STEP_7B, name="rising", num_q_heads=64, num_kv_heads=8, cache_len=0, num_new=900, input_scale=0.3, seed=61)
    x = W.make_step_inputs(cfg)
    _rising_scores(x["q_new"], x["k_new"], [0], [900])
    r = oracle_step("bf16", x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], 0, cfg.rope_theta)
    for fused in (False, True):
        gs = GpuStep(handle, "bf16", 64, 8, 128, 900, cfg.rope_theta, 900, fused=fused)
        g = gs.step(0, x["q_new"], x["k_new"], x["v_new"])
        check_output("bf16", g["out"], g["lse"], r["out"], r["lse"])


def test_references_move_in_later_items_of_a_paged_batch(handle):
    new = [450, 300, 470, 140, 431, 260]
    cfg = dataclasses.replace(W.PAGED_B16, name="rising", num_q_heads=64, num_kv_heads=8, batch=len(new), seed=62)
    x = W.make_paged_inputs(cfg, [0] * len(new), new)
    _rising_scores(x["q_new"], x["k_new"], x["new_offsets"], new)
    out, lse, k_pool, v_pool = _gpu_paged(handle, cfg, x)
    okp, ovp = f64(x["k_pool"]), f64(x["v_pool"])
    ref_out, ref_lse = so.step_paged(f64(x["q_new"]), f64(x["k_new"]), f64(x["v_new"]), okp, ovp, x["page_table"], [0] * len(new),
                                     x["new_offsets"], cfg.rope_theta, storage="bf16")
    check_output("bf16", out, lse, ref_out, ref_lse)
    _check_pools(x, cfg, k_pool, v_pool, okp, ovp)
