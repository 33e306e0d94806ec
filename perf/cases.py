"""The work this library is used for, as timed cases: layer passes over video streams of every size, the same kernels in
full-causal mode, decode steps, a live stream, a video with a shorter last block, and a batch with multimodal positions.

Every case goes through the public entry points (`layer.py`, `binding.py`) the way a caller strings them together.
Inputs are N(0, 1) in bf16, as the pre-RoPE Q, K, V of the synthetic workloads; `outliers` scales the first four sink K
rows by 8 (the attention-sink feature of real key caches).  Caches that a case starts from hold keys as they are after
RoPE, which keeps the distribution.
"""
import math

import torch

from paper_2506_19651_b200 import binding as pb
from paper_2506_19651_b200.layer import LayerBuffers, StreamingWindow, layer_forward, ragged_layer_forward

MROPE_SECTIONS = {128: (16, 24, 24), 64: (8, 12, 12)}
FRAME = 256  # tokens of one frame (16 x 16 patches) in the multimodal position ids


def _case(kind, S, B, N, Q, Hq, Hkv, d=128, theta=1e6, outliers=True, last=0, batch=1, name=None):
    c = {"kind": kind, "S": S, "B": B, "N": N, "Q": Q, "Hq": Hq, "Hkv": Hkv, "d": d, "theta": theta, "outliers": outliers,
         "last": last, "batch": batch}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a clip of a few frames through a small model: launches and host time count
        _case("layer", 64, 128, 4, 32, 4, 2, d=64, theta=1e4, outliers=False, name="layer_tiny"),
        # 64 frames, 12.6K tokens: an ordinary video question
        _case("layer", 784, 784, 15, 64, 28, 4, name="layer_12k"),
        # 50K tokens: a long video
        _case("layer", 1568, 1568, 31, 128, 28, 4, name="layer_50k"),
        # one layer of the 74K-token stack, with a long question
        _case("layer", 1152, 1152, 63, 256, 28, 4, name="layer_74k"),
        # the block-size sweep's ends: one frame a block, 32 frames a block
        _case("layer", 256, 256, 127, 64, 32, 8, outliers=False, name="layer_blocks_256"),
        _case("layer", 8192, 8192, 3, 64, 32, 8, outliers=False, name="layer_blocks_8192"),
        # heads of 64
        _case("layer", 1024, 1024, 15, 64, 32, 8, d=64, outliers=False, name="layer_head64"),
        # plain causal attention by the same calls: what the block mask is compared with
        _case("causal", 784, 784, 15, 64, 28, 4, name="causal_12k"),
        # one generated token against the resident cache of the long video
        _case("decode", 1568, 1568, 31, 1, 28, 4, name="decode_50k"),
        # a live stream: one new block of 784 tokens into a window of 8, then a question of 24 tokens
        _case("stream", 784, 784, 8, 24, 28, 4, name="stream_step"),
        # a video that does not divide evenly: odd sizes everywhere, buffers allocated by the call
        _case("ragged", 777, 1000, 12, 37, 14, 2, last=431, name="ragged_video"),
        # two sequences in one call each, positions by (time, height, width)
        _case("mrope", 512, 1024, 7, 40, 28, 4, batch=2, name="mrope_batch2"),
    ]


def _between(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    most = {k: max(work(c)[k] for c in listed()) for k in ("bytes", "flops")}
    while True:
        kind = rng.choice(["layer"] * 6 + ["causal", "decode", "decode", "stream", "ragged", "mrope"])
        d = 64 if rng.random() < 0.2 else 128
        Hq, Hkv = rng.choice([(28, 4), (28, 4), (32, 8), (14, 2), (8, 2), (4, 2)])
        tokens = _between(rng, 448, 74000 if kind != "causal" else 14000)
        B = _between(rng, 64, min(8192, max(64, tokens // 2)))
        if rng.random() < 0.6:
            B = max(64, B // 16 * 16)  # whole patches, as frames come
        S = B if rng.random() < 0.6 else _between(rng, 16, 4096)
        N = max(1, (tokens - S) // B)
        Q = _between(rng, 1, 256)
        last, batch = 0, 1
        if kind == "decode":
            Q = rng.choice([1, 1, 1, 2, 4, 8])
        elif kind == "stream":
            N, Q = rng.choice([2, 4, 8, 16]), _between(rng, 1, 64)
        elif kind == "ragged":
            N, last = N + 1, rng.randint(1, B - 1)
        elif kind == "mrope":
            batch = rng.choice([1, 2, 3, 4])
            N = max(1, N // batch)
        c = _case(kind, S, B, N, Q, Hq, Hkv, d=d, outliers=rng.random() < 0.6, last=last, batch=batch)
        w = work(c)
        if w["bytes"] <= most["bytes"] and w["flops"] <= most["flops"]:
            return c


def _n_video(c):
    return c["S"] + c["N"] * c["B"] if not c["last"] else c["S"] + (c["N"] - 1) * c["B"] + c["last"]


def _shape(c):
    return pb.make_shape(c["S"], c["B"], c["N"], c["Q"], c["Hq"], c["Hkv"], c["d"], theta=c["theta"], batch=c["batch"],
                         mask_mode=pb.MASK_FULL_CAUSAL if c["kind"] == "causal" else pb.MASK_PEVLM)


def _triangle(n):
    return n * (n + 1) // 2


def work(c):
    """Bytes: un-roped Q, K, V read once, the caches, outputs and LSE written once (for a decode or stream step the resident
    cache is read too).  FLOPs: 4 d Hq for every visible (query, key) pair."""
    S, B, N, Q, Hq, Hkv, d = (c[k] for k in ("S", "B", "N", "Q", "Hq", "Hkv", "d"))
    nv = _n_video(c)
    q_row, kv_row, lse_row = Hq * d * 2, 2 * Hkv * d * 2, Hq * 4
    if c["kind"] == "decode":
        pairs = Q * nv + _triangle(Q)
        rows, resident = Q, nv
    elif c["kind"] == "stream":
        pairs = B * S + _triangle(B) + Q * nv + _triangle(Q)
        rows, resident = B + Q, nv  # the question reads sink and window, the new block's rows among them
    else:
        pairs = Q * nv + _triangle(Q)
        if c["kind"] == "causal":
            pairs += _triangle(nv)
        else:
            pairs += _triangle(S) + sum(b * S + _triangle(b) for b in [B] * (N - 1 if c["last"] else N) + ([c["last"]] if c["last"] else []))
        rows, resident = nv + Q, 0
    b = rows * (2 * q_row + 2 * kv_row + lse_row) + resident * kv_row
    return {"bytes": c["batch"] * b, "flops": c["batch"] * 4 * d * Hq * pairs}


def tolerance(c):
    """bf16 outputs of sums over bf16 probabilities.  Against 64-bit arithmetic on the same roped bf16 inputs the outputs are
    off by 1.5e-3 (12.6K tokens; 1.5e-3 of it is the rounding of the result to bf16) to 2.2e-3 (tiny layer, rows of few
    keys), single values by at most 4e-2 of the root mean square, LSE by 1e-7: about four times the first, twice the second."""
    return {"rel": 0.008, "max": 0.08}


def _normal(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).to(torch.bfloat16)


def _qkv(c, gen, n):
    q, k, v = _normal(gen, n, c["Hq"], c["d"]), _normal(gen, n, c["Hkv"], c["d"]), _normal(gen, n, c["Hkv"], c["d"])
    return q, k, v


def _positions3(n_video, Q):
    """(time, height, width) of every token: a grid of patches for each frame, then the question's running index."""
    i = torch.arange(n_video, device="cuda", dtype=torch.int32)
    side = int(math.isqrt(FRAME))
    video = torch.stack([i // FRAME, i % FRAME // side, i % side])
    start = max(n_video // FRAME + 1, side)
    question = torch.arange(start, start + Q, device="cuda", dtype=torch.int32).repeat(3, 1)
    return video.contiguous(), question.contiguous()


def prepare(c, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, batch = c["kind"], c["batch"]
    S, B, N, Q, Hq, Hkv, d = (c[k] for k in ("S", "B", "N", "Q", "Hq", "Hkv", "d"))
    nv = _n_video(c)
    st = {"c": c}
    if kind in ("layer", "causal", "ragged"):
        st["qkv"] = _qkv(c, gen, nv + Q)
        if c["outliers"]:
            st["qkv"][1][:min(4, S)] *= 8
        if kind != "ragged":
            st["buf"] = LayerBuffers(_shape(c))
    elif kind == "decode":
        s = st["shape"] = _shape(c)
        st["q"], st["k"], st["v"] = _qkv(c, gen, Q)
        st["k_cache"], st["v_cache"] = _normal(gen, nv + Q, Hkv, d), _normal(gen, nv + Q, Hkv, d)
        if c["outliers"]:
            st["k_cache"][:min(4, S)] *= 8
        st["q_roped"], st["o"] = torch.empty_like(st["q"]), torch.empty_like(st["q"])
        st["lse"] = torch.empty((Hq, Q), dtype=torch.float32, device="cuda")
        st["ws"] = torch.zeros(pb.pevlm_workspace_bytes(s, pb.WS_QUERY), dtype=torch.uint8, device="cuda")
    elif kind == "stream":
        win = st["win"] = StreamingWindow(S, B, N, max(Q, 1), Hq, Hkv, d, c["theta"])
        q, k, v = _qkv(c, gen, S)
        if c["outliers"]:
            k[:min(4, S)] *= 8
        win.set_sink(q, k, v)
        for _ in range(N):
            win.append_block(*_qkv(c, gen, B))
        st["seen"] = win.blocks_seen
        st["block"], st["question"] = _qkv(c, gen, B), _qkv(c, gen, Q)
    else:  # mrope: the video rows and the question rows of all sequences, each kind in a tensor of its own
        s = st["shape"] = _shape(c)
        st["video"], st["question"] = _qkv(c, gen, batch * nv), _qkv(c, gen, batch * Q)
        if c["outliers"]:
            for b in range(batch):
                st["video"][1][b * nv:b * nv + min(4, S)] *= 8
        pos_v, pos_q = _positions3(nv, Q)
        st["pos_v"], st["pos_q"] = pos_v.repeat(batch, 1, 1), pos_q.repeat(batch, 1, 1)
        st["roped"] = [torch.empty_like(t) for t in st["video"][:2] + st["question"][:2]]
        st["k_cache"] = torch.empty((batch * (nv + Q), Hkv, d), dtype=torch.bfloat16, device="cuda")
        st["v_cache"] = torch.empty_like(st["k_cache"])
        st["o_v"], st["o_q"] = torch.empty_like(st["video"][0]), torch.empty_like(st["question"][0])
        st["lse_v"] = torch.empty((batch, Hq, nv), dtype=torch.float32, device="cuda")
        st["lse_q"] = torch.empty((batch, Hq, Q), dtype=torch.float32, device="cuda")
        st["ws"] = [torch.zeros(pb.pevlm_workspace_bytes(s, w), dtype=torch.uint8, device="cuda") for w in (pb.WS_PREFILL, pb.WS_QUERY)]
    return st


def run(st):
    c = st["c"]
    kind, nv, Q = c["kind"], _n_video(c), c["Q"]
    if kind in ("layer", "causal"):
        b = layer_forward(st["buf"], *st["qkv"])
        return [b.o_video, b.lse_video, b.o_question, b.lse_question, b.k_cache, b.v_cache]
    if kind == "ragged":
        return ragged_layer_forward(*st["qkv"], c["S"], c["B"], c["N"], c["last"], Q, c["theta"])[:4]
    if kind == "decode":
        s = st["shape"]
        pb.pevlm_rope_qk(s, st["q"], st["k"], st["q_roped"], st["k_cache"][nv:], nv, Q)
        pb.pevlm_assemble_kv(s, None, None, None, st["v"], st["k_cache"], st["v_cache"])
        pb.pevlm_query_attn(s, st["q_roped"], st["k_cache"], st["v_cache"], st["o"], st["lse"], st["ws"])
        return [st["o"], st["lse"], st["k_cache"], st["v_cache"]]
    if kind == "stream":
        win = st["win"]
        win.blocks_seen = st["seen"]  # every pass is the same step of the stream: positions and slot do not run on
        return win.append_block(*st["block"]) + win.ask(*st["question"]) + (win.k_cache, win.v_cache)
    s, sections = st["shape"], MROPE_SECTIONS[c["d"]]
    (q_v, k_v, v_v), (q_q, k_q, v_q) = st["video"], st["question"]
    rq_v, rk_v, rq_q, rk_q = st["roped"]
    pb.pevlm_rope_qk_mrope(s, q_v, k_v, rq_v, rk_v, nv, st["pos_v"], sections)
    pb.pevlm_rope_qk_mrope(s, q_q, k_q, rq_q, rk_q, Q, st["pos_q"], sections)
    pb.pevlm_assemble_kv(s, rk_v, v_v, rk_q, v_q, st["k_cache"], st["v_cache"])
    pb.pevlm_parallel_prefill_attn(s, rq_v, rk_v, v_v, st["o_v"], st["lse_v"], st["ws"][0])
    pb.pevlm_query_attn(s, rq_q, st["k_cache"], st["v_cache"], st["o_q"], st["lse_q"], st["ws"][1])
    return [st["o_v"], st["lse_v"], st["o_q"], st["lse_q"], st["k_cache"], st["v_cache"]]
