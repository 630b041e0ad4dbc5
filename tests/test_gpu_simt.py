"""The SIMT step attention (float FMAs) at the edges of its tiles (128- and 32-row blocks, 64-key tiles)
against the fp64 oracle: the gates of the fp32 configuration (1e-5 on outputs and log-sum-exps).  fp32 takes it when
the caller asks for it; the same cases run on the kernels that fp32 takes by itself, whose row blocks and key tiles are alike."""
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


KERNELS = pytest.mark.parametrize("kernel", [B.EVLN_KERNEL_SIMT, B.EVLN_KERNEL_AUTO])


@KERNELS
@pytest.mark.parametrize("dtype,hq,hkv,d,L,n,splits", [
    ("f32", 2, 1, 64, 0, 1, 0),            # one key, one row per head
    ("f32", 1, 1, 128, 63, 1, 1),          # exactly one key tile
    ("f32", 4, 2, 64, 64, 16, 2),          # 32 rows: one small block; the new keys start a tile
    ("f32", 3, 1, 128, 200, 11, 0),        # 33 rows, ragged keys
    ("f32", 28, 4, 128, 700, 196, 0),      # 128-row blocks, the last one partly filled
    ("f32", 28, 4, 128, 1024, 128, 1),     # long serial walk, no split
    ("f32", 8, 4, 64, 2000, 64, 32),       # the most splits
    ("f32", 2, 2, 64, 10, 3, 7),           # more splits than key tiles (splits of one or two keys)
    ("f32", 14, 2, 128, 5, 300, 3),        # mostly causal: whole key ranges invisible to early rows
    ("bf16", 14, 2, 64, 321, 70, 0),       # bf16 of head_dim 64 runs here too
    ("bf16", 28, 4, 64, 1500, 196, 0),
    ("f32", 28, 4, 128, 1024, 196, 0),     # equal shares of the key tiles, each over the end of a row block
    ("f32", 8, 1, 64, 5000, 64, 0),        # ... of two or three tiles: a row in many parts
    ("f32", 7, 1, 128, 40, 1170, 0),       # ... of the most row blocks, short ones first
    ("f32", 7, 1, 64, 40, 1172, 0),        # one row block more: no shares
])
def test_simt_step_against_oracle(handle, dtype, hq, hkv, d, L, n, splits, kernel):
    # unit-variance inputs in fp32 (softmax far from uniform); 0.3 in bf16, where the operands' rounding
    # scales with the logits and is not what is tested here
    cfg = W.StepConfig("simt", dtype, hq, hkv, d, L, n, 1e4, 1.0 if dtype == "f32" else 0.3, 40 + L + n)
    x = W.make_step_inputs(cfg)
    gs = GpuStep(handle, dtype, hq, hkv, d, L + n + 5, cfg.rope_theta, n, num_splits=splits, kernel=kernel)
    gs.load_cache(x["k_cache"], x["v_cache"])
    g = gs.step(L, x["q_new"], x["k_new"], x["v_new"])
    r = oracle_step(dtype, x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], L, cfg.rope_theta)
    check_cache(gs, r, L, n)
    check_output(dtype, g["out"], g["lse"], r["out"], r["lse"])


@KERNELS
@pytest.mark.parametrize("dtype,hq,hkv,d,L,n", [
    ("f32", 2, 1, 64, 100, 20),            # 32-row blocks
    ("f32", 28, 4, 128, 1024, 196),        # equal shares of 128-row blocks
    ("f32", 8, 8, 64, 0, 700),             # several key tiles that rows of the same block see in part
    ("bf16", 14, 2, 64, 321, 70),
])
def test_values_of_keys_a_row_does_not_see(handle, dtype, hq, hkv, d, L, n, kernel):
    # infinite and undefined values at token `bad` reach the rows of the tokens from `bad` on, and no others
    cfg = W.StepConfig("unseen", dtype, hq, hkv, d, L, n, 1e4, 1.0 if dtype == "f32" else 0.3, 90 + L + n)
    x = W.make_step_inputs(cfg)
    r = oracle_step(dtype, x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], L, cfg.rope_theta)
    bad = n * 2 // 3
    v = x["v_new"].clone()
    v[bad, :, :d // 2] = float("inf")
    v[bad, :, d // 2:] = float("nan")
    gs = GpuStep(handle, dtype, hq, hkv, d, L + n + 5, cfg.rope_theta, n, kernel=kernel)
    gs.load_cache(x["k_cache"], x["v_cache"])
    g = gs.step(L, x["q_new"], x["k_new"], v)
    check_output(dtype, g["out"][:bad], g["lse"][:bad], r["out"][:bad], r["lse"][:bad])
    assert not bool(torch.isfinite(g["out"][bad:]).any())
