"""What this library is used for, as cases that can be timed: generated tokens (xq_decode_step), prompts and pieces of
prompts going into the cache (xq_append_kv), and several query tokens at once (xq_append_kv, then xq_attention_chunk).

Shapes are those of the repository's workloads (paper_2510_11236_b200/workloads.py), of its tests, or generic.  A cache
grows with every pass; one whose room is used up starts over with its prompt, as a server's does with the next
request.  Keys, values and queries follow the recipe of workloads.py: N(0, 1), outlier key channels, the second layer
of a pair close to the first.
"""
from __future__ import annotations

import math

import torch

import paper_2510_11236_b200 as xq

ETA1, ETA2 = 1.0 / 6.0, 0.045  # calibration parameters of the paper's main results
INPUT_SETS = 4                 # new tokens and queries that a step cycles through


def _case(name, kind, *, layers, batch, q_heads, kv_heads, context, tokens=1, room, head_dim=128, group=32,
          residual=128, kq=None, vq=None, f16=False, host=False, share_group=0, gamma1=0.0):
    return dict(name=name, kind=kind, layers=layers, batch=batch, q_heads=q_heads, kv_heads=kv_heads,
                head_dim=head_dim, context=context, tokens=tokens, room=room, group=group, residual=residual,
                kq=layers if kq is None else kq, vq=layers if vq is None else vq, f16=f16, host=host,
                share_group=share_group, gamma1=gamma1)


def listed():
    return [
        # a tiny layer pair (head_dim 64, 512 tokens): a call's own overhead
        _case("step_tiny_pair", "step", layers=2, batch=1, q_heads=4, kv_heads=4, head_dim=64, context=512, room=2048,
              residual=32),
        # one user, a short chat: 32 layers, 1000 tokens, 2-bit keys and 1-bit values
        _case("step_one_user_1k", "step", layers=32, batch=1, q_heads=32, kv_heads=8, context=1000, room=4096, vq=0),
        # every query head with its own kv head, batch 8, 4k context, 2-bit keys and values
        _case("step_mha_4k", "step", layers=32, batch=8, q_heads=32, kv_heads=32, context=4096, room=4096),
        # the headline: groups of four query heads, batch 4, 32k context, 2-bit keys, 1-bit values
        _case("step_gqa_32k", "step", layers=32, batch=4, q_heads=32, kv_heads=8, context=32768, room=4096, vq=0),
        # quantization groups of 64, window of 64, batch 16, 8k context, IEEE half precision
        _case("step_gqa_8k_g64", "step", layers=32, batch=16, q_heads=32, kv_heads=8, context=8192, room=4096,
              group=64, residual=64, f16=True),
        # one sequence of 128k tokens
        _case("step_long_128k", "step", layers=32, batch=1, q_heads=32, kv_heads=8, context=131072, room=4096, vq=0),
        # groups of five query heads, 48 layers, the upper half of the values in 1 bit, inputs and results in pinned
        # host memory
        _case("step_group5_16k_host", "step", layers=48, batch=4, q_heads=40, kv_heads=8, context=16384, room=4096,
              vq=24, host=True),
        # whole prompts of a batch into the cache
        _case("append_prompt_4k", "append", layers=4, batch=8, q_heads=32, kv_heads=32, context=0, tokens=4096,
              room=4096),
        # one sequence's prompt in ragged pieces, layer by layer; the second layer of a pair merges its codes
        _case("append_pieces_merged", "append", layers=16, batch=1, q_heads=32, kv_heads=8, context=1024, tokens=333,
              room=16 * 333, vq=0, gamma1=0.4),
        # a few tokens at once behind a long context (drafted tokens to verify)
        _case("chunk_16_at_32k", "chunk", layers=4, batch=4, q_heads=32, kv_heads=8, context=32768, tokens=16,
              room=4096, vq=0),
        # a piece of a long prompt, ragged
        _case("chunk_250_at_8k", "chunk", layers=2, batch=1, q_heads=32, kv_heads=8, context=8192, tokens=250,
              room=16 * 250, vq=0),
        # the paper's timing workload (Appendix D): a prompt of 1024 tokens, whole
        _case("prompt_1024", "chunk", layers=2, batch=1, q_heads=32, kv_heads=32, context=0, tokens=1024, room=1024),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "append", "append", "chunk", "chunk"])
    head_dim = 64 if rng.random() < 0.1 else 128
    kv_heads = rng.choice([1, 2, 4, 8, 8, 8, 16, 32])
    q_heads = kv_heads * rng.choice([1, 2, 3, 4, 4, 5, 7, 8] if head_dim == 128 else [1, 3, 4])
    group = rng.choice([32, 32, 64]) if head_dim == 128 else 32
    residual = rng.choice([64, 128, 128, 256])
    batch = _log_int(rng, 1, 32)
    layers = 2 * _log_int(rng, 1, 16)
    gamma1 = 0.0
    share_group = 0
    # (sequence, kv head) streams x tokens of a layer: up to a million, fewer where no tensor-core kernel serves
    most = 1_000_000 if head_dim == 128 else 30_000
    if kind == "step":
        context = max(16, min(_log_int(rng, 64, 131072), most // (batch * kv_heads)))
        tokens, room = 1, 4096
        if rng.random() < 0.2:
            layers, share_group = 4 * max(1, layers // 4), 4
    elif kind == "append":
        layers = min(layers, 8)
        context = rng.choice([0, _log_int(rng, 16, 4096)])
        tokens = max(1, min(_log_int(rng, 1, 8192), 500_000 // (batch * kv_heads)))
        room = min(16, max(1, 16384 // tokens)) * tokens
        if rng.random() < 0.2:
            gamma1 = rng.choice([0.2, 0.4, 0.6])
    else:
        layers = 2
        if head_dim == 64:  # short pieces of a small model
            batch, kv_heads, q_heads = 1, 4, 4
        batch = min(batch, 8)
        tokens = _log_int(rng, 2, 512)
        # every query token reads everything before it: bounded by tokens x streams x context
        context = rng.choice([0, _log_int(rng, 64, 65536)])
        context = min(context, 60_000_000 // (layers * tokens * batch * kv_heads))
        room = 8 * tokens
    kq = rng.choice([layers, layers, layers // 2 if share_group == 0 and (layers // 2) % 2 == 0 else 0])
    vq = rng.choice([0, 0, layers])
    case = _case("", kind, layers=layers, batch=batch, q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim,
                 context=context, tokens=tokens, room=room, group=group, residual=residual, kq=kq, vq=vq,
                 f16=rng.random() < 0.25, host=kind == "step" and rng.random() < 0.2, share_group=share_group,
                 gamma1=gamma1)
    del case["name"]
    return case


def _config(c):
    return xq.make_config(n_layers=c["layers"], batch=c["batch"], n_q_heads=c["q_heads"], n_kv_heads=c["kv_heads"],
                          head_dim=c["head_dim"], max_seq=c["context"] + c["room"], group_size=c["group"],
                          residual_len=c["residual"], kq=c["kq"], vq=c["vq"], eta1=ETA1, eta2=ETA2,
                          io_dtype=xq.XQ_F16 if c["f16"] else xq.XQ_BF16, share_group=c["share_group"],
                          gamma1=c["gamma1"])


def _keys_values(c, gen, tokens):
    """K and V of a layer pair: [2][batch, kv_heads, tokens, head_dim] each."""
    dtype = torch.float16 if c["f16"] else torch.bfloat16
    shape = (c["batch"], c["kv_heads"], tokens, c["head_dim"])
    mult = torch.ones(c["kv_heads"], c["head_dim"], device="cuda")
    for h in range(c["kv_heads"]):
        mult[h, torch.randperm(c["head_dim"], generator=gen, device="cuda")[:3]] = 10.0
    k0 = torch.randn(shape, generator=gen, device="cuda").mul_(mult[None, :, None, :]).to(dtype)
    v0 = torch.randn(shape, generator=gen, device="cuda").to(dtype)
    near = [(x + 0.1 * torch.randn(shape, generator=gen, device="cuda")).to(dtype) for x in (k0, v0)]
    return [k0, near[0]], [v0, near[1]]


def _regions(cache, c, which):
    """The bytes of one kind of region of every layer, as few views of the workspace as their spacing allows."""
    n = c["batch"] * c["kv_heads"]
    period = c["share_group"] or 2
    views = []
    for first in range(period):
        place = []
        for layer in range(first, c["layers"], period):
            rc, offset, stride = xq.xq_region(cache.handle, layer, which)
            assert rc == 0
            place.append((offset, stride))
        while place:
            run = 1
            step = place[1][0] - place[0][0] if len(place) > 1 else 0
            while run < len(place) and place[run][1] == place[0][1] and place[run][0] - place[run - 1][0] == step:
                run += 1
            if place[0][1]:
                views.append(torch.as_strided(cache.workspace, (run, n * place[0][1]), (step, 1), place[0][0]))
            place = place[run:]
    return views


def _fill(state):
    c, cache = state["case"], state["cache"]
    if c["context"]:
        for layer in range(c["layers"]):
            cache.append_kv(layer, state["prompt"][0][layer % 2], state["prompt"][1][layer % 2])


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dtype = torch.float16 if c["f16"] else torch.bfloat16
    cache = xq.Cache(_config(c))
    cache.workspace.zero_()  # what no token has reached reads as zero
    state = dict(case=c, cache=cache, turn=0)
    state["prompt"] = _keys_values(c, gen, c["context"]) if c["context"] else None
    _fill(state)
    L, B, D = c["layers"], c["batch"], c["head_dim"]
    if c["kind"] == "step":
        sets = []
        for _ in range(INPUT_SETS):
            k, v = _keys_values(c, gen, L)  # one token for each layer
            k = [k[layer % 2][:, :, layer:layer + 1] for layer in range(L)]
            v = [v[layer % 2][:, :, layer:layer + 1] for layer in range(L)]
            q = torch.randn(L, B, c["q_heads"], D, generator=gen, device="cuda").to(dtype)
            new = [torch.stack(k).contiguous(), torch.stack(v).contiguous(), q]
            sets.append([t.cpu().pin_memory() for t in new] if c["host"] else new)
        state["new"] = sets
        state["out"] = torch.empty_like(sets[0][2]).pin_memory() if c["host"] else torch.empty_like(sets[0][2])
        state["window"] = [_regions(cache, c, which) for which in (4, 5)]
    else:
        state["new"] = _keys_values(c, gen, c["tokens"])
        if c["kind"] == "append":
            # codes, scales and zero-points, windows; a borrowing layer's codes are its owner's
            state["regions"] = [_regions(cache, c, which) for which in range(6)]
        else:
            state["q"] = torch.randn(2, c["tokens"], B, c["q_heads"], D, generator=gen, device="cuda").to(dtype)
            state["out"] = [torch.empty_like(state["q"][0]) for _ in range(L)]
    torch.cuda.synchronize()
    return state


def run(state):
    c, cache = state["case"], state["cache"]
    if cache.seq_len(c["layers"] - 1) + c["tokens"] > cache.cfg.max_seq:  # the next request
        cache.reset()
        _fill(state)
    if c["kind"] == "step":
        k, v, q = state["new"][state["turn"] % INPUT_SETS]
        state["turn"] += 1
        cache.decode_step(k, v, q, state["out"], mem=xq.XQ_MEM_HOST if c["host"] else xq.XQ_MEM_DEVICE)
        if c["host"]:
            torch.cuda.current_stream().synchronize()  # before the host may read the result
        return [state["out"], state["window"]]
    k, v = state["new"]
    for layer in range(c["layers"]):
        cache.append_kv(layer, k[layer % 2], v[layer % 2])
        if c["kind"] == "chunk":
            cache.attention_chunk(layer, state["q"][layer % 2], out=state["out"][layer])
    return state["regions"] if c["kind"] == "append" else state["out"]


def _packed_bytes(c, tokens):
    """Bytes of `tokens` quantized tokens of all layers: codes once for each sharing group, scale and zero-point of
    every layer."""
    streams, D, g = c["batch"] * c["kv_heads"], c["head_dim"], c["group"]
    period = c["share_group"] or 2
    codes = sum((2 if layer < c["kq"] else 1) + (2 if layer < c["vq"] else 1) for layer in range(0, c["layers"], period))
    return streams * tokens * (codes * D / 8 + c["layers"] * (4 * D / g + 4 * D / g))


def work(case):
    c = case
    L, streams, D, T = c["layers"], c["batch"] * c["kv_heads"], c["head_dim"], c["tokens"]
    S = c["context"] + T
    window = (S - 1) % c["residual"] + 1
    new = 4 * L * streams * T * D  # K and V of the new tokens, 16-bit
    if c["kind"] == "append":
        old_window = ((c["context"] - 1) % c["residual"] + 1) if c["context"] else 0
        packed = S - window - (c["context"] - old_window)
        moved = old_window if packed else 0  # window tokens that are read and quantized
        return {"bytes": new + 4 * L * streams * D * (moved + (window if packed else T)) + _packed_bytes(c, packed),
                "flops": 0}
    seen = sum(range(S - T + 1, S + 1))  # tokens that the query tokens attend to
    io = 4 * L * T * c["batch"] * c["q_heads"] * D
    return {"bytes": new + io + _packed_bytes(c, S - window) + 4 * L * streams * window * D + new,
            "flops": 4 * L * c["batch"] * c["q_heads"] * D * seen}


def tolerance(case):
    if case["kind"] == "append":
        return "exact"
    # The result's own rounding: two correct implementations differ by single units in the last place.  Measured, the
    # tensor-core kernel against the scalar fp32 one on the step cases: rel 1.8e-3 (bf16) and 6e-4 (f16), largest
    # difference 8e-3 of the value (one unit of bf16); stated are about four times that.
    return {"rel": 2e-3, "max": 0.03} if case["f16"] else {"rel": 6e-3, "max": 0.03}
