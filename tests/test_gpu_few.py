"""Steps of few rows (at most 32 packed query rows per kv head): the kernel that keeps its products in
registers and merges a head's blocks through their cluster, alone, as the one-launch step and on a page
pool, at the edges of its tiles (64-key stages, rings of stages, 16-row tiles, cluster shares)."""
import dataclasses

import pytest
import torch

from oracle import step_oracle as so
from paper_2512_10310_b200 import binding as B
from paper_2512_10310_b200 import workloads as W
from tests.helpers import GpuStep, check_cache, check_output, f64, oracle_step
from tests.test_gpu_paged import _check_pools, _gpu_paged

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handle():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    h = B.evlnCreate(0)
    yield h
    B.evlnDestroy(h)


@pytest.mark.parametrize("hq,hkv,L,n,splits", [
    (28, 4, 0, 1, 0),             # one key
    (28, 4, 63, 1, 0),            # exactly one stage
    (28, 4, 64, 2, 0),            # the new tokens start a stage; 14 rows
    (28, 4, 62, 4, 0),            # they straddle two stages of different blocks; 28 rows = two row tiles
    (4, 4, 1000, 16, 0),          # one query head per kv head, the most tokens of a fused step
    (2, 2, 700, 17, 0),           # one more: the three launches
    (32, 8, 5000, 4, 0),          # 16 rows, eight kv heads
    (64, 8, 3000, 4, 0),          # 32 rows: the most
    (64, 8, 3068, 4, 0),          # 32 rows over a longer cache of eight kv heads: the one-CTA kernel
    (28, 4, 9000, 3, 0),          # more stages per block than the ring holds
    (7, 1, 20000, 1, 0),          # one kv head: the library splits
    (6, 6, 25000, 17, 0),         # 17 rows over a long cache of six kv heads: the one-CTA kernel
    (64, 8, 4292, 4, 1),          # 32 rows of eight kv heads in fewer splits than fill the SMs: clusters do
    (28, 4, 500, 1, 5),           # splits of one and two stages: clusters of one block
    (28, 4, 100, 1, 9),           # more splits than stages: empty splits
])
def test_step_of_few_rows_against_oracle(handle, hq, hkv, L, n, splits):
    cfg = W.StepConfig("few", "bf16", hq, hkv, 128, L, n, 1e6, 0.3, 700 + L + n)
    x = W.make_step_inputs(cfg)
    r = oracle_step("bf16", x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], L, cfg.rope_theta)
    bits = []
    for fused in (True, False):
        gs = GpuStep(handle, "bf16", hq, hkv, 128, L + n + 3, cfg.rope_theta, n, num_splits=splits, fused=fused)
        gs.load_cache(x["k_cache"], x["v_cache"])
        g = gs.step(L, x["q_new"], x["k_new"], x["v_new"])
        check_cache(gs, r, L, n)
        check_output("bf16", g["out"], g["lse"], r["out"], r["lse"])
        bits.append((g["out"].view(torch.int16), g["lse"], g["q_rot"].reshape(-1).view(torch.int16), gs.k_cache.view(torch.int16)))
    for a, b in zip(*bits):
        assert torch.equal(a, b)


@pytest.mark.parametrize("hq,hkv,L,n", [
    (64, 8, 4292, 4),             # 32 rows of eight kv heads: the one-CTA kernel
    (28, 4, 24600, 4),            # 28 rows of four, from 24576 keys on
    (28, 4, 24600, 3),            # ... 21 rows: the few-row kernel
    (28, 4, 20000, 4),            # ... and below
    (28, 4, 4292, 8),             # 56 rows
    (28, 4, 4096, 196),           # CTA pairs
])
def test_reported_split_count_passed_on_gives_the_same_bits(handle, hq, hkv, L, n):
    gen = torch.Generator(device="cuda:0").manual_seed(L + n)
    q, k, v = (torch.randn((n, h, 128), generator=gen, device="cuda:0").to(torch.bfloat16) for h in (hq, hkv, hkv))
    kc, vc = (torch.randn((hkv, L, 128), generator=gen, device="cuda:0").to(torch.bfloat16) for _ in range(2))
    bits, splits = [], 0
    for _ in range(2):
        gs = GpuStep(handle, "bf16", hq, hkv, 128, L + n, 1e6, n, num_splits=splits, fused=True)
        gs.k_cache[:, :L], gs.v_cache[:, :L] = kc, vc
        g = gs.step(L, q, k, v)
        splits = g["splits"]
        bits.append((g["out"].view(torch.int16), g["lse"]))
    assert all(torch.equal(a, b) for a, b in zip(*bits))


@pytest.mark.parametrize("lens,new,chunk", [
    ([300, 64, 1], [1, 1, 1], 0),                 # shorter than a stage, one page, one key
    ([1000, 127, 128, 4000], [4, 2, 0, 3], 0),    # ragged, an episode without new tokens, two row tiles
    ([2500, 700], [1, 2], 4),                     # work items of the caller's size
    ([2500, 700], [4, 1], 16),                    # ... long ones of two row tiles: CTA pairs
    ([2500, 700], [4, 1], 24),                    # ... unsplit
    ([2500, 700] * 10, [4, 1] * 10, 16),          # ... more of them than pairs: the few-row kernel
])
def test_paged_batch_of_few_rows_against_oracle(handle, lens, new, chunk):
    cfg = dataclasses.replace(W.PAGED_B16, batch=len(lens), seed=60 + len(lens))
    x = W.make_paged_inputs(cfg, lens, new)
    out, lse, k_pool, v_pool = _gpu_paged(handle, cfg, x, kv_chunk_tiles=chunk)
    okp, ovp = f64(x["k_pool"]), f64(x["v_pool"])
    ref_out, ref_lse = so.step_paged(f64(x["q_new"]), f64(x["k_new"]), f64(x["v_new"]), okp, ovp, x["page_table"], lens,
                                     x["new_offsets"], cfg.rope_theta, storage="bf16")
    check_output("bf16", out, lse, ref_out, ref_lse)
    _check_pools(x, cfg, k_pool, v_pool, okp, ovp)
