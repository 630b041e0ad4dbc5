"""Buffers that a caller shares between the arguments of one call (rotation in place, the output over a buffer the call
has done with): the same bits as with buffers of their own, whatever the launches of the call do side by side."""
import dataclasses

import pytest
import torch

from paper_2512_10310_b200 import binding as B
from paper_2512_10310_b200 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
HQ, HKV, D = 28, 4, 128


@pytest.fixture(scope="module")
def handle():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    h = B.evlnCreate(0)
    yield h
    B.evlnDestroy(h)


def _step(handle, L, n, place):
    """One evlnStep; place(q, k, v, q_rot, out) says where the tensors of the call lie."""
    cfg = dataclasses.replace(W.STEP_7B, name="shared", cache_len=L, num_new=n, seed=50 + L + n)
    x = W.make_step_inputs(cfg)
    p = B.step_params("bf16", HQ, HKV, D, L, n, L + n, cfg.rope_theta)
    kc, vc = (torch.zeros((HKV, L + n, D), dtype=torch.bfloat16, device=DEV) for _ in range(2))
    kc[:, :L] = x["k_cache"].to(DEV).permute(1, 0, 2)
    vc[:, :L] = x["v_cache"].to(DEV).permute(1, 0, 2)
    fresh = lambda *s: torch.full(s, 3.0, dtype=torch.bfloat16, device=DEV)
    q, k, v, q_rot, out = place(fresh(n, HQ, D), fresh(n, HKV, D), fresh(n, HKV, D), fresh(n, HQ, D), fresh(n, HQ, D))
    for t, src in ((q, "q_new"), (k, "k_new"), (v, "v_new")):
        t.copy_(x[src].to(DEV))
    ws = torch.empty(B.evlnStepWorkspaceSize(handle, p), dtype=torch.uint8, device=DEV)
    lse = torch.zeros((n, HQ), dtype=torch.float32, device=DEV)
    B.evlnStep(handle, p, q, k, v, q_rot, kc, vc, ws, out, lse)
    assert B.evlnGetDeviceStatus(handle) == 0
    return out.view(torch.int16).clone(), lse, kc.view(torch.int16), vc.view(torch.int16)


def _in_projection(q, k, v, q_rot, out):
    """q, k, v as views of one [n, Hq + 2 Hkv, D] buffer that the output is then laid over."""
    n = q.shape[0]
    qkv = torch.full((n, HQ + 2 * HKV, D), 3.0, dtype=torch.bfloat16, device=DEV)
    return qkv[:, :HQ], qkv[:, HQ:HQ + HKV], qkv[:, HQ + HKV:], q_rot, qkv.view(-1)[:n * HQ * D].view(n, HQ, D)


@pytest.mark.parametrize("L,n,place", [
    (4292, 1, lambda q, k, v, r, o: (q, k, v, q, o)),        # one token rotated in place
    (4292, 1, lambda q, k, v, r, o: (q, k, v, r, r)),        # the output over the rotated queries
    (4292, 4, lambda q, k, v, r, o: (q, k, v, r, q)),        # ... over the queries
    (700, 4, _in_projection),                                # ... over queries, keys and values of other tokens
    (0, 256, lambda q, k, v, r, o: (q, k, v, r, r)),         # unsplit on CTA pairs, units that start late
    (500, 1100, lambda q, k, v, r, o: (q, k, v, r, r)),      # ... more of them than pairs
    (4096, 196, lambda q, k, v, r, o: (q, k, v, r, r)),      # split
], ids=["q_rot=q", "out=q_rot", "out=q", "out=qkv", "unsplit", "persistent", "split"])
def test_step_on_shared_buffers(handle, L, n, place):
    want = _step(handle, L, n, lambda *t: t)
    for a, b in zip(_step(handle, L, n, place), want):
        assert torch.equal(a, b)


def test_allocation_free_call_over_its_queries(handle):
    p = B.step_params("bf16", HQ, HKV, D, 0, 256, 256, 1e6)
    assert B.evlnStepNumSplits(handle, p) == 1
    gen = torch.Generator(device=DEV).manual_seed(9)
    kc, vc = (torch.randn((HKV, 256, D), generator=gen, device=DEV).to(torch.bfloat16) for _ in range(2))
    q_rot = torch.randn((256 * HQ * D,), generator=gen, device=DEV).to(torch.bfloat16)
    out = torch.empty_like(q_rot)
    B.evlnStepAttentionNoAlloc(p, q_rot, kc, vc, out)
    B.evlnStepAttentionNoAlloc(p, q_rot, kc, vc, q_rot)
    assert B.evlnGetDeviceStatus(None) == 0
    assert torch.equal(q_rot.view(torch.int16), out.view(torch.int16))
