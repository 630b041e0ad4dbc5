"""Short unsplit steps on one CTA per 128-row tile, on both sides of where that form begins, against the fp64 oracle; one call and
three give the same bits."""
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


@pytest.mark.parametrize("hq,hkv,L,n", [
    (28, 4, 0, 18),        # 126 rows: one tile
    (28, 4, 0, 19),        # 133: five rows in the second
    (28, 4, 0, 256),
    (28, 4, 316, 196),     # 512 keys: the most key tiles
    (28, 4, 317, 196),     # one more: CTA pairs
    (64, 8, 0, 288),       # 18 tiles of 8 heads: the most
    (64, 8, 0, 289),       # one more: CTA pairs
    (8, 8, 100, 200),      # tiles that end with a token's rows
])
def test_short_unsplit_steps(handle, hq, hkv, L, n):
    cfg = W.StepConfig("single", "bf16", hq, hkv, 128, L, n, 1e6, 0.3, 70 + L + n)
    x = W.make_step_inputs(cfg)
    r = oracle_step("bf16", x["k_cache"], x["v_cache"], x["q_new"], x["k_new"], x["v_new"], L, cfg.rope_theta)
    got = []
    for fused in (False, True):
        gs = GpuStep(handle, "bf16", hq, hkv, 128, L + n + 5, cfg.rope_theta, n, num_splits=1, fused=fused)
        gs.load_cache(x["k_cache"], x["v_cache"])
        g = gs.step(L, x["q_new"], x["k_new"], x["v_new"])
        check_cache(gs, r, L, n)
        check_output("bf16", g["out"], g["lse"], r["out"], r["lse"])
        got.append(g)
    assert torch.equal(got[0]["out"], got[1]["out"]) and torch.equal(got[0]["lse"], got[1]["lse"])
