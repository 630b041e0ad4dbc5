"""The work that users of this library have it do, as cases that can be timed and compared.

A case is a dict of plain values; its "kind" says which entry points it goes through:

  step     one model step on contiguous caches: every layer rotates and appends the new tokens and
           attends over its own cache (evlnStep, or the three calls one by one)
  paged    the same for a batch of episodes on page pools
  packed   a packed sequence under the action-isolating mask (evlnPackedForward)
  reindex  a step on an un-rotated store: the new frame goes to the store, a sampler picks the history
           frames, the kept segments are laid out and rotated, then the step runs on the result

"layers" is how many transformer layers a pass goes through; each has caches of its own, as in a
model, so that a pass of many layers finds its caches in device memory rather than in L2.
"""
import math

import torch

from paper_2512_10310_b200 import binding as B

DEV = "cuda:0"
THETA = {"bf16": 1.0e6, "f32": 1.0e4}
TORCH_DTYPE = {"bf16": torch.bfloat16, "f32": torch.float32}
PAGE = 64
HEADS_7B = {"q_heads": 28, "kv_heads": 4, "head_dim": 128}
HEADS_70B = {"q_heads": 64, "kv_heads": 8, "head_dim": 128}


def listed():
    step = {"kind": "step", "dtype": "bf16", "table": True, "calls": 1, "lse": False}
    return [
        # the smallest call: the single-layer fp32 step that numerics are checked on (64 instruction
        # tokens + 3 frames of 64 cached, one new frame)
        {**step, "name": "tiny_f32_step", "dtype": "f32", "q_heads": 2, "kv_heads": 1, "head_dim": 64, "layers": 1,
         "cached": 256, "new": 64, "table": False, "lse": True},
        # a layer of the 7B-class model in fp32: the precision reference that a bf16 deployment is held against
        {**step, **HEADS_7B, "name": "f32_layer", "dtype": "f32", "layers": 1, "cached": 1024, "new": 196, "table": False,
         "lse": True},
        # one action token decoded after a frame, through a whole 28-layer model
        {**step, **HEADS_7B, "name": "action_token", "layers": 28, "cached": 4292, "new": 1},
        # a chunk of action tokens at the end of a 100-step episode, whole model
        {**step, **HEADS_7B, "name": "action_chunk_late", "layers": 28, "cached": 20656, "new": 8},
        # the instruction at the start of an episode: prefill on an empty cache, whole model
        {**step, **HEADS_7B, "name": "instruction_prefill", "layers": 28, "cached": 0, "new": 256},
        # the new-frame step of one layer through the three calls (a program that puts its own work between them)
        {**step, **HEADS_7B, "name": "frame_three_calls", "layers": 1, "cached": 4096, "new": 196, "table": False,
         "calls": 3, "lse": True},
        # the 50th frame of a streaming episode (196 visual + 8 action tokens), whole model
        {**step, **HEADS_7B, "name": "stream_frame", "layers": 28, "cached": 10252, "new": 204},
        # a long history on the 70B-class head shape
        {**step, **HEADS_70B, "name": "long_history_70b", "layers": 1, "cached": 32768, "new": 256, "table": False},
        # serving 16 concurrent episodes of ragged lengths: a new frame for each ...
        {"kind": "paged", **HEADS_7B, "name": "paged_frames", "layers": 1, "batch": 16, "shortest": 1024, "longest": 16384,
         "new_least": 196, "new_most": 196, "table": True},
        # ... and an action token for each
        {"kind": "paged", **HEADS_7B, "name": "paged_action_tokens", "layers": 4, "batch": 16, "shortest": 1024,
         "longest": 16384, "new_least": 1, "new_most": 1, "table": True},
        # forward pass over a packed sequence: instruction, then 12 frames with their action chunks
        {"kind": "packed", **HEADS_7B, "name": "packed_sequence", "layers": 1, "instruction": 256, "frame": 196, "action": 8,
         "frames": 12},
        # the un-rotated store at its 64th frame, the uniform sampler keeps 16 frames, whole model
        {"kind": "reindex", **HEADS_7B, "name": "reindexed_step", "layers": 28, "instruction": 256, "frame": 196, "frames": 64,
         "budget": 16, "sampler": B.EVLN_SAMPLE_UNIFORM, "stride": 1},
    ]


# ---- drawn cases ---------------------------------------------------------------------------

def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    kind = rng.choice(["f32", "tokens", "prefill", "frame", "frame", "long", "paged", "paged", "packed", "reindex"])
    heads = rng.choice([HEADS_7B, HEADS_7B, HEADS_70B, {"q_heads": 32, "kv_heads": 8, "head_dim": 128}])
    layers = _log_int(rng, 1, 28)
    step = {"kind": "step", "dtype": "bf16", **heads, "layers": layers, "table": rng.random() < 0.5,
            "calls": rng.choice([1, 1, 3]), "lse": rng.random() < 0.3}
    if kind == "f32":
        kv = rng.choice([1, 2, 4])
        return {**step, "dtype": "f32", "q_heads": kv * rng.choice([1, 2, 4, 7]), "kv_heads": kv,
                "head_dim": rng.choice([64, 128]), "layers": 1, "cached": _log_int(rng, 64, 2048), "new": _log_int(rng, 8, 256)}
    if kind == "tokens":
        return {**step, "cached": _log_int(rng, 256, 32768), "new": _log_int(rng, 1, 16)}
    if kind == "prefill":
        return {**step, "cached": 0, "new": _log_int(rng, 32, 1024)}
    if kind == "frame":
        return {**step, "cached": _log_int(rng, 256, 32768), "new": rng.randint(64, 256)}
    if kind == "long":
        return {**step, "layers": rng.choice([1, 2]), "cached": _log_int(rng, 16384, 65536), "new": rng.randint(128, 256)}
    if kind == "paged":
        frames = rng.random() < 0.5
        longest = _log_int(rng, 1024, 16384)
        return {"kind": "paged", **heads, "layers": rng.choice([1, 2, 4]), "batch": _log_int(rng, 2, 32),
                "shortest": max(1, longest // rng.choice([2, 4, 16])), "longest": longest,
                "new_least": 64 if frames else 1, "new_most": 256 if frames else rng.choice([1, 4, 8, 16]),
                "table": rng.random() < 0.5}
    if kind == "packed":
        return {"kind": "packed", **heads, "layers": rng.choice([1, 2, 4]), "instruction": rng.randint(32, 400),
                "frame": rng.choice([64, 196, rng.randint(32, 256)]), "action": rng.randint(1, 16), "frames": _log_int(rng, 2, 24)}
    return {"kind": "reindex", **heads, "layers": layers, "instruction": rng.randint(64, 400), "frame": rng.randint(64, 256),
            "frames": _log_int(rng, 4, 64), "budget": rng.choice([8, 16, 16]),
            "sampler": rng.choice([B.EVLN_SAMPLE_UNIFORM, B.EVLN_SAMPLE_SLIDING]), "stride": rng.choice([1, 2, 4])}


def draw(rng):
    most = [work(c) for c in listed()]
    most_bytes, most_flops = max(w["bytes"] for w in most), max(w["flops"] for w in most)
    most_f32 = max(work(c)["flops"] for c in listed() if c.get("dtype") == "f32")
    while True:
        c = _draw_once(rng)
        w = work(c)
        flops_limit = most_f32 if c.get("dtype") == "f32" else most_flops
        if w["bytes"] <= most_bytes and w["flops"] <= flops_limit:
            return c


# ---- lengths that follow from a case ---------------------------------------------------------

def _paged_lens(c):
    """Cache lengths spread evenly over [shortest, longest] and new-token counts over [new_least, new_most]: ragged,
    not aligned to anything, the same for every seed (the seed deals the pages and draws the values)."""
    b = c["batch"]
    lens = [c["shortest"] + (c["longest"] - c["shortest"]) * ((7 * i + 3) % b) // max(b - 1, 1) - (i % 3 if c["shortest"] > 3 else 0)
            for i in range(b)]
    new = [c["new_least"] + (c["new_most"] - c["new_least"]) * ((5 * i + 1) % b) // max(b - 1, 1) for i in range(b)]
    return lens, new


def _kept_frames(c):
    """How many history frames the sampler keeps."""
    if c["sampler"] == B.EVLN_SAMPLE_UNIFORM:
        return min(c["frames"], c["budget"])
    return min((c["frames"] - 1) // c["stride"] + 1, c["budget"])


def _causal_pairs(cached, new):
    return new * cached + new * (new + 1) // 2


def work(case):
    """Each input read once and each output written once; 4 * head_dim operations per visible (query, key) pair and query head."""
    c = case
    hq, hkv, d, layers = c["q_heads"], c["kv_heads"], c["head_dim"], c["layers"]
    eb = 4 if c.get("dtype") == "f32" else 2
    q_row, kv_row = hq * d * eb, 2 * hkv * d * eb             # one token's queries (or outputs); its keys and values
    if c["kind"] == "step":
        n, pairs = c["new"], _causal_pairs(c["cached"], c["new"])
        # cache read, queries in, outputs out, new keys and values in and appended
        size = c["cached"] * kv_row + 2 * n * q_row + 2 * n * kv_row + (4 * n * hq if c["lse"] else 0)
    elif c["kind"] == "paged":
        lens, new = _paged_lens(c)
        pairs = sum(_causal_pairs(a, b) for a, b in zip(lens, new))
        size = sum(lens) * kv_row + sum(new) * 2 * (q_row + kv_row)
    elif c["kind"] == "packed":
        vis = c["instruction"] + c["frames"] * c["frame"]
        act = c["frames"] * c["action"]
        pairs = _causal_pairs(0, vis)
        pairs += sum(_causal_pairs(c["instruction"] + (t + 1) * c["frame"], c["action"]) for t in range(c["frames"]))
        # the sequence in, outputs out, the cache of the visual tokens written
        size = (vis + act) * (2 * q_row + kv_row) + vis * kv_row
    else:
        kept = c["instruction"] + _kept_frames(c) * c["frame"]
        pairs = _causal_pairs(kept, c["frame"])
        # new frame in, stored and appended; the kept tokens read and laid out; queries in, outputs out
        size = 3 * c["frame"] * kv_row + 2 * kept * kv_row + 2 * c["frame"] * q_row
    return {"bytes": layers * size, "flops": layers * 4 * d * hq * pairs}


def tolerance(case):
    # fp32: sums of 32-bit products.  bf16: one rounding of the probabilities and one of the result.
    if case.get("dtype") == "f32":
        return {"rel": 1e-5, "max": 2e-4}
    return {"rel": 1e-2, "max": 5e-2}


# ---- what a program has in hand before the pass ------------------------------------------------

_handle = None


def _the_handle():
    """One handle for the process, as a program keeps it."""
    global _handle
    if _handle is None:
        torch.cuda.set_device(0)
        _handle = B.evlnCreate(0)
    return _handle


def _randn(gen, shape, dtype):
    return torch.randn(shape, generator=gen, device=DEV, dtype=dtype)


def _bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device=DEV)


def _params(c, cached, new, capacity, s):
    return B.step_params(c.get("dtype", "bf16"), c["q_heads"], c["kv_heads"], c["head_dim"], cached, new, capacity,
                         THETA[c.get("dtype", "bf16")], rope_table=s.get("table"),
                         rope_table_first_pos=s.get("table_first", 0), rope_table_count=s.get("table_count", 0))


def _qkv(gen, c, new, dtype, s):
    """Queries, keys and values of the new tokens as the three views of the projection's fused output."""
    hq, hkv, d = c["q_heads"], c["kv_heads"], c["head_dim"]
    qkv = _randn(gen, (c["layers"], new, hq + 2 * hkv, d), dtype)
    s["q"] = [x[:, :hq] for x in qkv]
    s["k"] = [x[:, hq:hq + hkv] for x in qkv]
    s["v"] = [x[:, hq + hkv:] for x in qkv]


def prepare(case, seed):
    c = case
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    h = _the_handle()
    layers, hq, hkv, d = c["layers"], c["q_heads"], c["kv_heads"], c["head_dim"]
    dtype = TORCH_DTYPE[c.get("dtype", "bf16")]
    s = {"case": c, "h": h}
    if c["kind"] == "step":
        n = c["new"]
        cap = c["cached"] + n
        s["kc"], s["vc"] = (_randn(gen, (layers, hkv, cap, d), dtype) for _ in range(2))
        s["kcs"], s["vcs"] = list(s["kc"]), list(s["vc"])
        _qkv(gen, c, n, dtype, s)
        s["out"] = torch.zeros((layers, n, hq, d), dtype=dtype, device=DEV)
        s["outs"] = list(s["out"])
        s["lse"] = torch.zeros((layers, n, hq), dtype=torch.float32, device=DEV) if c["lse"] else None
        s["lses"] = list(s["lse"]) if c["lse"] else [None] * layers
        if c["table"]:
            s["table"] = _bytes(B.evlnRopeTableBytes(d, n))
            s["table_first"], s["table_count"] = c["cached"], n
        p = _params(c, c["cached"], n, cap, s)
        s["cap"] = cap
        s["q_rot"] = _bytes(B.evlnStepQRotSize(h, p))
        s["ws"] = _bytes(B.evlnStepWorkspaceSize(h, p))
    elif c["kind"] == "paged":
        lens, new = _paged_lens(c)
        need = [(a + b + PAGE - 1) // PAGE for a, b in zip(lens, new)]
        pages, total = sum(need) + 8, sum(new)
        deal = torch.randperm(pages, generator=gen, device=DEV).tolist()
        rows, at = [], 0
        for k in need:
            rows.append(deal[at:at + k] + [0] * (max(need) - k))
            at += k
        s["pages"], s["row"] = pages, max(need)
        s["lens"], s["offsets"] = lens, [0]
        for k in new:
            s["offsets"].append(s["offsets"][-1] + k)
        s["page_table"] = torch.tensor(rows, dtype=torch.int32, device=DEV)
        s["kc"], s["vc"] = (_randn(gen, (layers, pages, hkv, PAGE, d), dtype) for _ in range(2))
        s["kcs"], s["vcs"] = list(s["kc"]), list(s["vc"])
        s["q"], s["k"], s["v"] = (list(_randn(gen, (layers, total, m, d), dtype)) for m in (hq, hkv, hkv))
        s["out"] = torch.zeros((layers, total, hq, d), dtype=dtype, device=DEV)
        s["outs"] = list(s["out"])
        if c["table"]:
            s["table_first"], s["table_count"] = 0, max(lens) + max(new)
            s["table"] = _bytes(B.evlnRopeTableBytes(d, s["table_count"]))
            B.evlnRopeTable(h, d, THETA["bf16"], 0, s["table_count"], s["table"])
        p = _paged_params(s)
        s["q_rot"] = _bytes(total * hq * d * 2)
        s["ws"] = _bytes(B.evlnPagedWorkspaceSize(h, p, s["lens"], s["offsets"]))
    elif c["kind"] == "packed":
        vis = c["instruction"] + c["frames"] * c["frame"]
        total = vis + c["frames"] * c["action"]
        s["kc"], s["vc"] = (torch.zeros((layers, hkv, vis, d), dtype=dtype, device=DEV) for _ in range(2))
        s["kcs"], s["vcs"] = list(s["kc"]), list(s["vc"])
        _qkv(gen, c, total, dtype, s)
        s["out"] = torch.zeros((layers, total, hq, d), dtype=dtype, device=DEV)
        s["outs"] = list(s["out"])
        s["cap"] = vis
        s["ws"] = _bytes(B.evlnPackedWorkspaceSize(h, _packed_params(s)))
    else:
        n = c["frame"]
        s["stored"] = c["instruction"] + c["frames"] * n               # the history; the new frame goes behind it
        s["store_cap"] = s["stored"] + n
        kept = c["instruction"] + _kept_frames(c) * n
        s["cap"] = kept + n
        s["ks"], s["vs"] = (_randn(gen, (layers, hkv, s["store_cap"], d), dtype) for _ in range(2))
        s["kss"], s["vss"] = list(s["ks"]), list(s["vs"])
        s["kc"], s["vc"] = (torch.zeros((layers, hkv, s["cap"], d), dtype=dtype, device=DEV) for _ in range(2))
        s["kcs"], s["vcs"] = list(s["kc"]), list(s["vc"])
        _qkv(gen, c, n, dtype, s)
        s["out"] = torch.zeros((layers, n, hq, d), dtype=dtype, device=DEV)
        s["outs"] = list(s["out"])
        # positions 0 .. capacity are the same in every step of the episode: one table for all of them
        s["table_first"], s["table_count"] = 0, s["cap"]
        s["table"] = _bytes(B.evlnRopeTableBytes(d, s["cap"]))
        B.evlnRopeTable(h, d, THETA["bf16"], 0, s["cap"], s["table"])
        p = _params(c, kept, n, s["cap"], s)
        s["q_rot"] = _bytes(B.evlnStepQRotSize(h, p))
        s["ws"] = _bytes(B.evlnStepWorkspaceSize(h, p))
    return s


def _paged_params(s):
    c = s["case"]
    return B.paged_params(c["q_heads"], c["kv_heads"], c["head_dim"], c["batch"], PAGE, s["pages"], s["row"], THETA["bf16"],
                          rope_table=s.get("table"), rope_table_first_pos=s.get("table_first", 0),
                          rope_table_count=s.get("table_count", 0))


def _packed_params(s):
    c = s["case"]
    return B.packed_params(c["q_heads"], c["kv_heads"], c["head_dim"], c["instruction"], c["frame"], c["action"], c["frames"],
                           s["cap"], THETA["bf16"])


# ---- one pass ----------------------------------------------------------------------------------

def _run_step(s):
    c, h = s["case"], s["h"]
    # the parameters (and the table of the step's positions) hold for all layers of the step
    p = _params(c, c["cached"], c["new"], s["cap"], s)
    if c["table"]:
        B.evlnRopeTable(h, c["head_dim"], THETA[c["dtype"]], c["cached"], c["new"], s["table"])
    for i in range(c["layers"]):
        if c["calls"] == 1:
            B.evlnStep(h, p, s["q"][i], s["k"][i], s["v"][i], s["q_rot"], s["kcs"][i], s["vcs"][i], s["ws"], s["outs"][i],
                       s["lses"][i])
        else:
            B.evlnRopeAppend(h, p, s["q"][i], s["k"][i], s["v"][i], s["q_rot"], s["kcs"][i], s["vcs"][i])
            B.evlnStepAttention(h, p, s["q_rot"], s["kcs"][i], s["vcs"][i], s["ws"])
            B.evlnStepCombine(h, p, s["ws"], s["outs"][i], s["lses"][i])
    return [s["out"], s["kc"], s["vc"]] + ([s["lse"]] if c["lse"] else [])


def _run_paged(s):
    h, lens, offsets, table = s["h"], s["lens"], s["offsets"], s["page_table"]
    p = _paged_params(s)
    for i in range(s["case"]["layers"]):
        B.evlnPagedRopeAppend(h, p, s["q"][i], s["k"][i], s["v"][i], lens, offsets, table, s["q_rot"], s["kcs"][i], s["vcs"][i])
        B.evlnPagedStepAttention(h, p, s["q_rot"], s["kcs"][i], s["vcs"][i], lens, offsets, table, s["ws"])
        B.evlnPagedStepCombine(h, p, s["ws"], lens, offsets, s["outs"][i])
    return [s["out"], s["kc"], s["vc"]]


def _run_packed(s):
    p = _packed_params(s)
    for i in range(s["case"]["layers"]):
        B.evlnPackedForward(s["h"], p, s["q"][i], s["k"][i], s["v"][i], s["kcs"][i], s["vcs"][i], s["ws"], s["outs"][i])
    return [s["out"], s["kc"], s["vc"]]


def _run_reindex(s):
    c, h = s["case"], s["h"]
    frames = B.evlnSampleFrames(c["sampler"], c["frames"], c["budget"], c["stride"])
    src = [0] + [c["instruction"] + f * c["frame"] for f in frames]
    length = [c["instruction"]] + [c["frame"]] * len(frames)
    g = B.gather_params("bf16", c["kv_heads"], c["head_dim"], s["store_cap"], s["cap"], THETA["bf16"], s["table"],
                        s["table_first"], s["table_count"])
    p = _params(c, sum(length), c["frame"], s["cap"], s)
    for i in range(c["layers"]):
        B.evlnStoreAppend(h, g, s["k"][i], s["v"][i], s["stored"], s["kss"][i], s["vss"][i])
        B.evlnGatherRope(h, g, src, length, s["kss"][i], s["vss"][i], s["kcs"][i], s["vcs"][i])
        B.evlnStep(h, p, s["q"][i], s["k"][i], s["v"][i], s["q_rot"], s["kcs"][i], s["vcs"][i], s["ws"], s["outs"][i])
    return [s["out"], s["kc"], s["vc"], s["ks"], s["vs"]]


def run(state):
    return {"step": _run_step, "paged": _run_paged, "packed": _run_packed, "reindex": _run_reindex}[state["case"]["kind"]](state)
