"""The fp32 step attention on the tensor cores (three bf16 parts per float) at the edges of its tiles, where
its splitting of numbers ends, and as one launch."""
import numpy as np
import pytest
import torch

from paper_2512_10310_b200 import binding as B
from paper_2512_10310_b200 import workloads as W
from tests.helpers import GpuStep, check_cache, check_output, f64, oracle_step

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handle():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    h = B.evlnCreate(0)
    yield h
    B.evlnDestroy(h)


def _inputs(hq, hkv, d, L, n):
    cfg = W.StepConfig("f32", "f32", hq, hkv, d, L, n, 1e4, 1.0, 20 + L + n)
    return cfg, W.make_step_inputs(cfg)


def _step(handle, cfg, x, **options):
    gs = GpuStep(handle, "f32", cfg.num_q_heads, cfg.num_kv_heads, cfg.head_dim, cfg.cache_len + cfg.num_new + 5, cfg.rope_theta,
                 cfg.num_new, **options)
    gs.load_cache(x["k_cache"], x["v_cache"])
    return gs, gs.step(cfg.cache_len, x["q_new"], x["k_new"], x["v_new"])


@pytest.mark.parametrize("hq,hkv,d,L,n,splits", [
    (1, 1, 64, 0, 1, 0),           # one row, one key
    (2, 1, 64, 256, 64, 0),        # 128 rows
    (1, 1, 128, 62, 2, 1),         # keys end with their tile
    (4, 2, 128, 63, 64, 0),        # ... and one key into the third
    (7, 1, 128, 300, 18, 4),       # 126 rows
    (43, 1, 64, 100, 3, 0),        # 129 rows: a row block of one row
    (8, 1, 128, 449, 63, 8),       # 512 keys, a tile per split
    (8, 1, 128, 450, 63, 8),       # ... and one key more
    (8, 1, 64, 1000, 24, 16),      # as many splits as a cluster takes
    (8, 1, 64, 1000, 24, 17),      # one more
    (2, 2, 64, 10, 3, 7),          # more splits than key tiles
    (2, 2, 128, 30, 16, 1),        # 16 rows: one row tile
    (3, 1, 128, 500, 11, 0),       # 33 rows: a block of one row
    (1, 1, 128, 100, 81, 1),       # angles of more tokens than a block holds
    (8, 4, 128, 0, 64, 0),         # no cache
    (8, 4, 128, 200, 65, 0),       # 130 rows per head
    (28, 4, 128, 1024, 196, 0),    # equal shares
])
def test_one_call_is_the_three_calls(handle, hq, hkv, d, L, n, splits):
    cfg, x = _inputs(hq, hkv, d, L, n)
    r = oracle_step("f32", x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], L, cfg.rope_theta)
    three, a = _step(handle, cfg, x, num_splits=splits)
    one, b = _step(handle, cfg, x, num_splits=splits, fused=True)
    for gs, g in ((three, a), (one, b)):
        check_cache(gs, r, L, n)
        check_output("f32", g["out"], g["lse"], r["out"], r["lse"])
    for key in ("out", "lse", "q_rot"):
        assert torch.equal(a[key], b[key]), key
    assert torch.equal(three.k_cache, one.k_cache) and torch.equal(three.v_cache, one.v_cache)


@pytest.mark.parametrize("hq,hkv,d,L,n,scale", [
    (2, 1, 64, 256, 64, 1e-36),    # the parts of such numbers are not exact: done again in floats
    (28, 4, 128, 1024, 196, 1e-37),
    (4, 2, 128, 500, 70, 1e-36),
    (4, 2, 128, 500, 70, 1e30),
])
@pytest.mark.parametrize("fused", [False, True])
def test_values_of_any_size(handle, hq, hkv, d, L, n, scale, fused):
    cfg, x = _inputs(hq, hkv, d, L, n)
    x["v_cache"], x["v_new"] = x["v_cache"] * scale, x["v_new"] * scale
    r = oracle_step("f32", x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], L, cfg.rope_theta)
    _, g = _step(handle, cfg, x, fused=fused)
    # (the output is linear in V: the fp32 gate, relative)
    assert np.linalg.norm(f64(g["out"]) / scale - r["out"] / scale) <= 1e-5 * np.linalg.norm(r["out"] / scale)


@pytest.mark.parametrize("hq,hkv,d,L,n", [(2, 1, 64, 256, 64), (4, 2, 128, 500, 70), (28, 4, 128, 1024, 196)])
@pytest.mark.parametrize("q_size,k_size,softmax_scale", [
    (1e-36, 1e36, 0.0),            # the queries' third parts are below bf16's least number, and the keys are as large
    (1e36, 1e-36, 0.0),
    (1e-30, 1e30, 0.0),            # all parts exact
    (2.0 ** -56, 2.0 ** -56, 2.0 ** 110),      # products of parts below the least float
    (1e-2, 1e-2, 1e3),
])
@pytest.mark.parametrize("fused", [False, True])
def test_queries_and_keys_of_any_size(handle, hq, hkv, d, L, n, q_size, k_size, softmax_scale, fused):
    cfg, x = _inputs(hq, hkv, d, L, n)
    x["q_new"] = x["q_new"] * q_size
    x["k_cache"], x["k_new"] = x["k_cache"] * k_size, x["k_new"] * k_size
    r = oracle_step("f32", x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], L, cfg.rope_theta, scale=softmax_scale)
    _, g = _step(handle, cfg, x, fused=fused, scale=softmax_scale)
    check_output("f32", g["out"], g["lse"], r["out"], r["lse"])


@pytest.mark.parametrize("hq,hkv,d,L,n", [(2, 1, 64, 256, 64), (4, 2, 128, 500, 70), (28, 4, 128, 1024, 196)])
def test_scores_beyond_any_sum(handle, hq, hkv, d, L, n):
    # one key so long that it either takes a row over or drops out of it, by the sign of one channel of the query
    cfg, x = _inputs(hq, hkv, d, L, n)
    x["k_cache"][L // 2] = 0.0
    x["k_cache"][L // 2, :, 3] = -1.0e37
    r = oracle_step("f32", x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], L, cfg.rope_theta)
    _, g = _step(handle, cfg, x)
    assert np.abs(f64(g["out"]) - r["out"]).max() <= 1e-5


def test_new_keys_rotated_in_place(handle):
    # one kv head: its new tokens can be given in the cache slots they are stored to.  80 rows: more than one block's
    hq, d, L, n = 4, 64, 100, 20
    cfg, x = _inputs(hq, 1, d, L, n)
    _, want = _step(handle, cfg, x, fused=True)
    dev = "cuda:0"
    p = B.step_params("f32", hq, 1, d, L, n, L + n, cfg.rope_theta)
    kc, vc = (torch.cat([x[a], x[b]]).permute(1, 0, 2).contiguous().to(dev) for a, b in (("k_cache", "k_new"), ("v_cache", "v_new")))
    q, out = x["q_new"].to(dev), torch.empty((n, hq, d), device=dev)
    q_rot = torch.empty(B.evlnStepQRotSize(handle, p), dtype=torch.uint8, device=dev)
    ws = torch.empty(B.evlnStepWorkspaceSize(handle, p), dtype=torch.uint8, device=dev)
    B.evlnStep(handle, p, q, kc[0, L:].view(n, 1, d), vc[0, L:].view(n, 1, d), q_rot, kc, vc, ws, out, None)
    assert torch.equal(out, want["out"])


@pytest.mark.parametrize("hq,hkv,d,L,n,splits,first,count", [
    (8, 1, 64, 1000, 24, 12, 768, 64),         # split 9 of 12; evlnStep in one launch
    (28, 4, 128, 1024, 196, 12, 960, 64),      # ... of 12, 128-row blocks
])
def test_infinite_values_of_keys_without_weight(handle, hq, hkv, d, L, n, splits, first, count):
    # `count` keys whose scores are 150 below all others: what they hold is not in the result, in one call or in three
    cfg, x = _inputs(hq, hkv, d, L, n)
    slow = d // 2 - 1                          # the channel that turns least: half a radian over these positions
    x["q_new"][:, :, slow] = 40.0
    x["q_new"][:, :, slow + d // 2] = 0.0
    keys = torch.cat([x["k_cache"], x["k_new"]])
    keys[:, :, slow] = 0.0
    keys[first:first + count, :, slow] = -80.0
    values = torch.cat([x["v_cache"], x["v_new"]])
    got = []
    for filler in (0.0, float("inf")):
        values[first:first + count] = filler
        y = dict(x, k_cache=keys[:L], k_new=keys[L:], v_cache=values[:L], v_new=values[L:])
        for fused in (False, True):
            got.append(_step(handle, cfg, y, num_splits=splits, fused=fused)[1]["out"])
    assert torch.equal(got[0], got[1]) and torch.equal(got[2], got[3])
    assert bool(torch.isfinite(got[2]).all()) and torch.equal(got[0], got[2])


@pytest.mark.parametrize("hq,hkv,d,n", [
    (64, 64, 64, 1),               # 32-row blocks
    (64, 64, 128, 1),
    (28, 4, 64, 400),              # 128-row blocks
    (28, 4, 128, 400),
])
@pytest.mark.parametrize("fused", [False, True])
def test_log_sum_exp_of_one_key(handle, hq, hkv, d, n, fused):
    # The first token on an empty cache is not turned and sees itself only.  Scores of short numbers are exact, so what is left is
    # one rounding of the scale's product and one of its rest: half a unit of the last place each.
    cfg, x = _inputs(hq, hkv, d, 0, n)
    for key in ("q_new", "k_new"):
        x[key] = torch.round(x[key] * 4.0) / 4.0
    x["q_new"][0, :, 5:] = 0.0                 # few channels: scores of every size from 1/16 on
    _, g = _step(handle, cfg, x, fused=fused)
    k = f64(x["k_new"][0]).repeat(hq // hkv, axis=0)
    want = (f64(x["q_new"][0]) * k).sum(-1) / np.sqrt(d)
    assert bool((np.abs(f64(g["lse"][0]) - want) <= 2.0 ** -23 * np.abs(want)).all())
    assert np.array_equal(f64(g["out"][0]), f64(x["v_new"][0]).repeat(hq // hkv, axis=0))


@pytest.mark.parametrize("hq,hkv,d,L,n", [
    (2, 1, 64, 256, 64),
    (8, 4, 128, 362, 79),
    (4, 2, 64, 858, 40),
    (28, 4, 64, 1024, 196),
    (28, 4, 128, 1024, 196),
    (16, 4, 128, 2031, 252),
])
@pytest.mark.parametrize("kind", ["normal", "positive", "short"])
def test_no_further_off_than_float_fmas(handle, hq, hkv, d, L, n, kind):
    # tensor-core and SIMT kernels on the same inputs, both against the oracle.  An error of thousands of outputs is steady
    # within some per cent from one seed to the next; a quarter is allowed.
    cfg, x = _inputs(hq, hkv, d, L, n)
    for key in ("q_new", "k_new", "k_cache", "v_new", "v_cache"):
        if kind == "positive" and key[0] != "v":
            x[key] = x[key].abs()
        if kind == "short":
            x[key] = torch.round(x[key] * 4.0) / 4.0
    r = oracle_step("f32", x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], L, cfg.rope_theta)
    off = []
    for kernel in (B.EVLN_KERNEL_SIMT, B.EVLN_KERNEL_AUTO):
        _, g = _step(handle, cfg, x, kernel=kernel)
        off.append((np.linalg.norm(f64(g["out"]) - r["out"]), np.linalg.norm(f64(g["lse"]) - r["lse"])))
    assert off[1][0] <= 1.25 * off[0][0] and off[1][1] <= 1.25 * off[0][1], off


@pytest.mark.parametrize("hq,hkv,d,L,n,first", [
    (2, 1, 64, 256, 64, 128),      # 32-row blocks
    (28, 4, 128, 1024, 196, 512),  # equal shares of 128-row blocks
    (28, 4, 64, 0, 400, 0),        # 128-row blocks, the first keys seen by all
])
@pytest.mark.parametrize("count,depth,value", [
    (1, 75.0, 1.0),
    (64, 88.0, 1000.0),            # a key tile whose weights are below the least normal number
])
def test_small_sums_of_ordinary_values(handle, hq, hkv, d, L, n, first, count, depth, value):
    # A channel whose only values are at keys of weights below 1e-33: as accurate as any, and the other channels are the bits
    # that they are with something else in it, so nothing was done again in floats for its sake.
    cfg, x = _inputs(hq, hkv, d, L, n)
    slow = d // 2 - 1                          # the channel that turns least
    x["q_new"][:, :, slow] = 40.0
    x["q_new"][:, :, slow + d // 2] = 0.0
    keys, values = torch.cat([x["k_cache"], x["k_new"]]), torch.cat([x["v_cache"], x["v_new"]])
    keys[:, :, slow] = 0.0
    keys[first:first + count] = 0.0
    keys[first:first + count, :, slow] = -depth * d ** 0.5 / 40.0
    outs = []
    for other in (1.0, 0.0):
        values[:, :, 5] = other
        values[first:first + count, :, 5] = value
        y = dict(x, k_cache=keys[:L], k_new=keys[L:], v_cache=values[:L], v_new=values[L:])
        outs.append(_step(handle, cfg, y)[1]["out"])
    r = oracle_step("f32", y["k_cache"], y["v_cache"], y["q_new"], y["k_new"], y["v_new"], L, cfg.rope_theta)
    rows = slice(count if L == 0 else 0, None)     # (the first tokens of an empty cache see those keys only)
    want, got = r["out"][rows, :, 5], f64(outs[1])[rows, :, 5]
    assert np.abs(want).max() < 1e-30
    # the weight's exponent is 75 to 95: a score of that size is some units of 2^-24 of itself off
    assert bool((np.abs(got - want) <= 4e-5 * np.abs(want)).all())
    keep = [c for c in range(d) if c != 5]
    assert torch.equal(outs[0][rows][:, :, keep], outs[1][rows][:, :, keep])
