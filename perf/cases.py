"""Timed cases of the framework: the calls a video model makes through its public entry points.

A case is one call (or the calls one token needs) on a handle that is in the
middle of a video: the arena, the weights and the inputs are in HBM, the
compressed state and the decode cache hold earlier frames.  Passes go on through
the video; when the decode cache is full the next video starts on the same
arena, as a program that serves one video after another does.

Inputs.  Q and K carry, per (stream, layer, KV head), a fixed direction along
which each key token has its own salience (log-weight N(0, 2^2)) and every query
looks, on top of unit noise: attention is concentrated and the same tokens stay
important from frame to frame, which is what the method assumes of a video (its
two assumptions, App. A).  V is N(0, 1).  The transformer block gets N(0, 1)
hidden states and N(0, 0.02^2) weights, and its own projections make Q and K.
"""
from __future__ import annotations

import math

import torch

from paper_2605_31598_gb300 import diagnostics
from paper_2605_31598_gb300.inputs import BLOCKS, BlockShape, Shape, block_weights
from paper_2605_31598_gb300.statekv import (SELECTION_IMPORTANCE, SELECTION_LAYER,
                                            SELECTION_RECENCY, StateKV, block_weights_array, check,
                                            make_config, statekv_block_config)

DEV = "cuda"
CYCLE = 3              # different frames that the timed passes take in turn
CACHE_BYTES = 6 << 30  # decode cache of a prefill case, at most (and at most 8192 frames)
SELECTION = {"importance": SELECTION_IMPORTANCE, "recency": SELECTION_RECENCY,
             "layer": SELECTION_LAYER}


def _prefill(name, hq, hkv, d, T, B, layers, streams=1, selection="importance", causal=True):
    return {"name": name, "kind": "prefill", "hq": hq, "hkv": hkv, "d": d, "T": T, "B": B,
            "layers": layers, "streams": streams, "selection": selection, "causal": causal}


def listed():
    return [
        # the toy stream: the smallest frame step, all launches and latency
        _prefill("prefill_toy", 4, 1, 64, 16, 32, 1),
        # one 7B layer, as a model calls the step from inside its decoder layer
        _prefill("prefill_7b_layer", 28, 4, 128, 196, 1568, 1),
        # a small backbone with head dim 64 and 259 tokens per frame: nothing is a multiple
        # of a tile, the pool (1259) not even of 4
        _prefill("prefill_ragged", 14, 2, 64, 259, 1000, 4),
        # the largest state of the paper's capacity sweep, at one 7B layer
        _prefill("prefill_16k_state", 28, 4, 128, 196, 16384, 1),
        # the 28-layer 7B stack in one call: the benchmark's workload
        _prefill("prefill_7b_stack", 28, 4, 128, 196, 2048, 28),
        # the 80-layer 72B stack: the largest call
        _prefill("prefill_72b_stack", 64, 8, 128, 196, 4096, 80),
        # exact full self-attention over 32 earlier frames (the baseline of every
        # wall-time figure; a prompt over the cache runs the same way)
        {"name": "full_attention_7b", "kind": "full", "hq": 28, "hkv": 4, "d": 128, "T": 196,
         "layers": 28, "history": 32, "scores": False},
        # one generated token through the 28 layers, one call per layer as a decoder
        # makes them, over a 64-frame video
        {"name": "decode_token_7b", "kind": "decode", "hq": 28, "hkv": 4, "d": 128, "T": 196,
         "layers": 28, "history": 64, "tokens": 1},
        # two 7B-width decoder layers around the step: one video, then eight per call
        {"name": "block_7b_1stream", "kind": "block", "hq": 28, "hkv": 4, "d": 128, "T": 196,
         "B": 2048, "layers": 2, "streams": 1, "hidden": 3584, "intermediate": 18944},
        {"name": "block_7b_8streams", "kind": "block", "hq": 28, "hkv": 4, "d": 128, "T": 196,
         "B": 2048, "layers": 2, "streams": 8, "hidden": 3584, "intermediate": 18944},
        # the assumption diagnostics of App. A: scores of a full-attention frame, then
        # concentration and state metrics of 128-frame score rows
        {"name": "scores_7b", "kind": "full", "hq": 28, "hkv": 4, "d": 128, "T": 196,
         "layers": 28, "history": 32, "scores": True},
        {"name": "diagnose_7b", "kind": "diagnose", "rows": 28, "n_hist": 25088, "T": 196, "B": 2048},
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    d = rng.choice([64, 128])
    hkv = rng.choice([1, 2, 4, 8])
    hq = hkv * rng.randint(1, 8)
    kind = rng.choice(["prefill"] * 5 + ["full", "decode", "block", "diagnose"])
    if kind == "prefill":
        T = _spread(rng, 16, 400)
        B = _spread(rng, 3 * T, 8192)  # room for the state to grow over a few frames
        layers, streams = _spread(rng, 1, 28), rng.choice([1, 1, 2, 4])
        c = _prefill("", hq, hkv, d, T, B, layers, streams,
                     rng.choice(["importance"] * 4 + ["recency", "layer"]), rng.random() < 0.8)
    elif kind == "full":
        c = {"kind": kind, "hq": hq, "hkv": hkv, "d": d, "T": _spread(rng, 16, 400),
             "layers": _spread(rng, 1, 28), "history": _spread(rng, 1, 40),
             "scores": rng.random() < 0.4}
    elif kind == "decode":
        c = {"kind": kind, "hq": hq, "hkv": hkv, "d": d, "T": _spread(rng, 49, 300),
             "layers": _spread(rng, 1, 28), "history": _spread(rng, 4, 128),
             "tokens": rng.choice([1, 1, 2])}
    elif kind == "block":
        c = {"kind": kind, "hq": hq, "hkv": hkv, "d": d, "T": _spread(rng, 32, 260),
             "B": _spread(rng, 1300, 4096), "layers": rng.randint(1, 3),
             "streams": rng.choice([1, 1, 2, 3, 5]), "hidden": 128 * _spread(rng, 4, 32),
             "intermediate": 8 * _spread(rng, 128, 2400)}
    else:
        T = _spread(rng, 16, 400)
        n = T * _spread(rng, 2, 128)
        c = {"kind": kind, "rows": _spread(rng, 1, 64), "n_hist": n, "T": T,
             "B": _spread(rng, 16, max(17, n))}
    c.pop("name", None)
    # never more than the largest listed case
    top = work(listed()[5])
    while c["kind"] == "prefill" and work(c)["flops"] > top["flops"]:
        c["layers"] = max(1, c["layers"] // 2)
    return c


# ------------------------------------------------------------------ shapes and inputs
def _shape(c, max_frames):
    return Shape(c["hq"], c["hkv"], c["d"], c["T"], c.get("B", c["T"]), max_frames,
                 num_layers=c["layers"], num_streams=c.get("streams", 1))


def _max_frames(c, fill):
    frame = 4 * c["streams"] * c["layers"] * c["hkv"] * c["T"] * c["d"]
    return max(fill + 16, min(8192, CACHE_BYTES // frame))


def _fill_frames(c):
    """Frames the handle has seen before the first pass.  Few heads: the state is full, and
    every pass evicts.  Many heads: the state is nearly full; it fills during the first
    passes, then every pass evicts."""
    full = c["B"] // c["T"]
    return full if c["streams"] * c["layers"] * c["hkv"] <= 8 else max(0, full - 2)


class _Video:
    """Q, K, V of one video's frames, frame after frame, from a seed."""

    def __init__(self, c, seed, tokens=None):
        self.c, self.T = c, tokens or c["T"]
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed))
        S, L, H, d = c.get("streams", 1), c["layers"], c["hkv"], c["d"]
        mu = self._n(S, L, 1, H, d).float()
        self.mu = (mu / mu.norm(dim=-1, keepdim=True)).to(torch.bfloat16)

    def _n(self, *shape):
        return torch.randn(shape, generator=self.g, device=DEV, dtype=torch.bfloat16)

    def frame(self, tokens=None):
        c, T = self.c, tokens or self.T
        S, L, H, G, d = c.get("streams", 1), c["layers"], c["hkv"], c["hq"] // c["hkv"], c["d"]
        q = self._n(S, L, T, H, G, d).add_(self.mu.unsqueeze(4), alpha=math.sqrt(d))
        k = self._n(S, L, T, H, d).add_(2.0 * self._n(S, L, T, H, 1) * self.mu)
        return q.view(S, L, T, H * G, d), k, self._n(S, L, T, H, d)


def _whole(eng, view):
    """All (stream, layer) of one of the handle's regions, from the view of the first."""
    c = eng.cfg
    off = view.data_ptr() - eng.arena.data_ptr()
    n = c.num_streams * c.num_layers
    return (eng.arena[off: off + n * view.numel() * view.element_size()].view(view.dtype)
            .view(c.num_streams, c.num_layers, *view.shape))


def _buffers(eng):
    k, v, pos, _ = eng.state(0, 0)
    ck, cv, _ = eng.cache(0, 0)
    return {"state_k": _whole(eng, k), "state_v": _whole(eng, v), "positions": _whole(eng, pos),
            "cache_k": _whole(eng, ck), "cache_v": _whole(eng, cv)}


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    return {"prefill": _prepare_prefill, "full": _prepare_full, "decode": _prepare_decode,
            "block": _prepare_block, "diagnose": _prepare_diagnose}[case["kind"]](case, seed)


def _run_frames(eng, video, n, out):
    for _ in range(n):
        q, k, v = video.frame()
        check(eng.prefill_frame(q, k, v, out), "prefill_frame")


def _prepare_prefill(c, seed):
    fill = _fill_frames(c)
    cfg = make_config(_shape(c, _max_frames(c, fill)), causal=c["causal"],
                      selection=SELECTION[c["selection"]])
    eng, video = StateKV(cfg), _Video(c, seed)
    S, L, H = c["streams"], c["layers"], c["hkv"]
    out = torch.zeros((S, L, c["T"], c["hq"], c["d"]), dtype=torch.bfloat16, device=DEV)
    imp = None
    if c["selection"] != "recency":
        imp = torch.zeros((S, L, H, c["B"] + c["T"]), device=DEV)
    _run_frames(eng, video, fill, out)
    frames = [video.frame() for _ in range(CYCLE)]
    torch.cuda.synchronize()
    return {"kind": c["kind"], "eng": eng, "frames": frames, "out": out, "imp": imp, "seen": fill, "at": 0,
            "results": {"out": out, "importance": imp, **_buffers(eng)}}


def _prepare_full(c, seed):
    eng, video = StateKV(make_config(_shape(c, c["history"] + 1))), _Video(c, seed)
    out = torch.zeros((1, c["layers"], c["T"], c["hq"], c["d"]), dtype=torch.bfloat16, device=DEV)
    _run_frames(eng, video, c["history"], out)
    s = {"kind": c["kind"], "eng": eng, "frames": [video.frame() for _ in range(CYCLE)], "out": out, "at": 0,
         "scores": None}
    if c["scores"]:
        s["scores"] = torch.zeros((1, c["layers"], (c["history"] + 1) * c["T"]), device=DEV)
        s["workspace"] = torch.empty(eng.scores_workspace_bytes(), dtype=torch.uint8, device=DEV)
    torch.cuda.synchronize()
    return s


def _decode_frames(c):
    return c["history"] + max(1, 16384 // c["T"])  # the video and room for its answer


def _prepare_decode(c, seed):
    eng, video = StateKV(make_config(_shape(c, _decode_frames(c)))), _Video(c, seed)
    out = torch.zeros((1, c["layers"], c["T"], c["hq"], c["d"]), dtype=torch.bfloat16, device=DEV)
    _run_frames(eng, video, c["history"], out)
    steps = []
    for _ in range(CYCLE):  # one contiguous q, k, v per layer
        q, k, v = video.frame(c["tokens"])
        steps.append([tuple(x[:, l:l + 1].contiguous() for x in (q, k, v)) for l in range(c["layers"])])
    outs = [torch.zeros_like(q) for q, _, _ in steps[0]]
    ck, cv, _ = eng.cache(0, 0)
    torch.cuda.synchronize()
    return {"kind": c["kind"], "case": c, "seed": seed, "eng": eng, "steps": steps, "outs": outs, "at": 0,
            "room": _decode_frames(c) * c["T"] - c["history"] * c["T"],
            "results": {"out": outs, "cache_k": _whole(eng, ck), "cache_v": _whole(eng, cv)}}


def _block_parts(c, seed):
    """Weights of every layer and the hidden states of the frames, in order."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) + 1)
    bs = BlockShape(c["hidden"], c["intermediate"], weight_std=BLOCKS["qwen7b"].weight_std)
    weights = block_weights(_shape(c, 1), bs, seed=int(seed), device=DEV)
    x = [torch.randn((c["streams"], c["T"], c["hidden"]), generator=g, device=DEV,
                     dtype=torch.bfloat16) for _ in range(2 + CYCLE)]
    return bs, weights, x


def _prepare_block(c, seed):
    bs, weights, x = _block_parts(c, seed)
    frame = 4 * c["streams"] * c["layers"] * c["hkv"] * c["T"] * c["d"]
    eng = StateKV(make_config(_shape(c, max(32, min(1024, CACHE_BYTES // frame)))))
    bc = statekv_block_config(bs.hidden, bs.intermediate, bs.rms_eps, bs.rope_theta, 1.0, 0)
    ws = torch.empty(eng.block_workspace_bytes(bc), dtype=torch.uint8, device=DEV)
    y, warr = torch.zeros_like(x[0]), block_weights_array(weights)
    for n in range(2):  # two frames of the video have gone through
        check(eng.block_frame(bc, warr, x[n], y, ws), "block_frame")
    torch.cuda.synchronize()
    return {"kind": c["kind"], "eng": eng, "bc": bc, "weights": weights, "warr": warr, "ws": ws, "x": x[2:], "y": y,
            "seen": 2, "at": 0, "results": {"out": y, **_buffers(eng)}}


def _diagnose_scores(c, seed):
    """Layer-level scores of two consecutive frames: attention masses, heavy-tailed, a
    token's mass much the same in both."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    stride = 2 * c["n_hist"] + c["T"]
    a = torch.randn((c["rows"], stride), generator=g, device=DEV) * 2.0
    b = a + 0.2 * torch.randn((c["rows"], stride), generator=g, device=DEV)
    return torch.exp(a), torch.exp(b)


def _prepare_diagnose(c, seed):
    now, nxt = _diagnose_scores(c, seed)
    torch.cuda.synchronize()
    return {"kind": c["kind"], "case": c, "now": now, "next": nxt}


# ------------------------------------------------------------------ run
def run(s):
    return {"prefill": _run_prefill, "full": _run_full, "decode": _run_decode, "block": _run_block,
            "diagnose": _run_diagnose}[s["kind"]](s)


def _next_video(s):
    """The cache is full: a new handle for the next video, on the same arena."""
    eng = s["eng"]
    torch.cuda.synchronize()
    cfg, arena = eng.cfg, eng.arena
    eng.close()
    s["eng"] = StateKV(cfg, arena=arena)


def _run_prefill(s):
    if s["seen"] == s["eng"].cfg.max_frames:
        _next_video(s)
        s["seen"] = 0
    q, k, v = s["frames"][s["at"] % CYCLE]
    check(s["eng"].prefill_frame(q, k, v, s["out"], s["imp"]), "prefill_frame")
    s["at"] += 1
    s["seen"] += 1
    return s["results"]


def _run_full(s):
    q, k, v = s["frames"][s["at"] % CYCLE]
    s["at"] += 1
    if s["scores"] is None:
        check(s["eng"].full_attention_frame(q, k, v, s["out"]), "full_attention_frame")
        return {"out": s["out"]}
    check(s["eng"].full_attention_scores(q, k, v, s["out"], s["scores"], s["workspace"]),
          "full_attention_scores")
    return {"out": s["out"], "scores": s["scores"]}


def _run_decode(s):
    c = s["case"]
    if s["room"] < c["tokens"]:
        _next_video(s)
        eng, video = s["eng"], _Video(c, s["seed"])
        out = torch.zeros((1, c["layers"], c["T"], c["hq"], c["d"]), dtype=torch.bfloat16, device=DEV)
        _run_frames(eng, video, c["history"], out)
        s["room"] = _decode_frames(c) * c["T"] - c["history"] * c["T"]
    step, eng = s["steps"][s["at"] % CYCLE], s["eng"]
    for l, (q, k, v) in enumerate(step):
        check(eng.decode_step(q, k, v, s["outs"][l], layer_begin=l, layer_count=1), "decode_step")
    s["at"] += 1
    s["room"] -= c["tokens"]
    return s["results"]


def _run_block(s):
    if s["seen"] == s["eng"].cfg.max_frames:
        _next_video(s)
        s["seen"] = 0
    check(s["eng"].block_frame(s["bc"], s["warr"], s["x"][s["at"] % CYCLE], s["y"], s["ws"]),
          "block_frame")
    s["at"] += 1
    s["seen"] += 1
    return s["results"]


def _run_diagnose(s):
    c = s["case"]
    n, T, B = c["n_hist"], c["T"], c["B"]
    return {"mask": diagnostics.topb_mask(s["now"], n, B),
            "concentration": diagnostics.concentration(s["now"], n, [max(1, B // 8), B]),
            **diagnostics.state_metrics(s["now"], s["next"], n, T, B)}


# ------------------------------------------------------------------ work
def _attention_flops(units, hq, d, T, before):
    return 4.0 * d * hq * units * (T * before + T * (T + 1) / 2)


def work(c):
    kind = c["kind"]
    if kind == "diagnose":
        # both score rows once, one mask out
        n = c["rows"] * (2 * c["n_hist"] + c["T"])
        return {"bytes": 4.0 * n + c["rows"] * (2 * c["n_hist"] + c["T"]), "flops": 2.0 * n}
    T, d, hq, hkv = c["T"], c["d"], c["hq"], c["hkv"]
    units = c["layers"] * c.get("streams", 1)
    if kind == "decode":
        n, rows = c["tokens"], c["history"] * T
        return {"bytes": 2.0 * units * d * (2 * hkv * (rows + 2 * n) + 2 * hq * n),
                "flops": _attention_flops(units, hq, d, n, rows)}
    frame = 2.0 * units * T * d * (2 * hq + 2 * hkv)  # Q, K, V in, O out
    if kind == "full":
        rows = c["history"] * T
        b = frame + 4.0 * units * hkv * d * rows
        if c["scores"]:
            b += 4.0 * units * (rows + T)
        return {"bytes": b, "flops": _attention_flops(units, hq, d, T, rows)}
    B = c["B"]
    state, cache = 4.0 * units * hkv * d * B, 4.0 * units * hkv * d * T
    step = _attention_flops(units, hq, d, T, B)
    if kind == "prefill":
        imp = 4.0 * units * hkv * (B + T) if c["selection"] != "recency" else 0.0
        return {"bytes": frame + state + cache + imp, "flops": step}
    H, I = c["hidden"], c["intermediate"]
    params = H * d * (2 * hq + 2 * hkv) + 3 * H * I
    return {"bytes": 2.0 * c["layers"] * params + state + cache + 4.0 * c["streams"] * T * H,
            "flops": step + 2.0 * units * T * params}


# ------------------------------------------------------------------ exact
def exact(case, seed):
    return {"prefill": _exact_prefill, "full": _exact_full, "decode": _exact_decode,
            "block": _exact_block, "diagnose": _exact_diagnose}[case["kind"]](case, seed)


def _attend(q, k, v, before, causal=True):
    """softmax(q k^T / sqrt(d)) v in 64 bits for q [T][Hq][d] and k, v [n][Hkv][d], of which
    the first `before` rows precede the frame, and the weight each key receives per KV head."""
    T, hq, d = q.shape
    n, hkv, _ = k.shape
    qh = q.double().view(T, hkv, hq // hkv, d).permute(1, 2, 0, 3).reshape(hkv, -1, d)
    kh, vh = k.double().transpose(0, 1), v.double().transpose(0, 1)
    z = torch.matmul(qh, kh.transpose(1, 2)).view(hkv, -1, T, n) / math.sqrt(d)
    if causal:
        t = torch.arange(T, device=q.device)
        z[..., before:] = z[..., before:].masked_fill(t[None, :] > t[:, None], -math.inf)
    p = torch.softmax(z, dim=-1)
    o = torch.matmul(p.view(hkv, -1, n), vh).view(hkv, -1, T, d)
    return o.permute(2, 0, 1, 3).reshape(T, hq, d), p.sum(dim=(1, 2))


def _exact_prefill(c, seed):
    fill, video, T, B = _fill_frames(c), _Video(c, seed), c["T"], c["B"]
    S, L, H = c["streams"], c["layers"], c["hkv"]
    past = [video.frame()[1:] for _ in range(fill)]  # all of them fit the state, in order
    q, k, v = video.frame()
    out = torch.zeros(q.shape, dtype=torch.float64, device=DEV)
    imp = torch.zeros((S, L, H, B + T), dtype=torch.float64, device=DEV)
    for s in range(S):
        for l in range(L):
            kk = torch.cat([p[0][s, l] for p in past] + [k[s, l]])
            vv = torch.cat([p[1][s, l] for p in past] + [v[s, l]])
            o, w = _attend(q[s, l], kk, vv, fill * T, c["causal"])
            out[s, l] = o
            imp[s, l, :, : fill * T] = w[:, : fill * T]
            imp[s, l, :, B:] = w[:, fill * T:]
    # the states and caches hold copies of input rows
    return {"out": out, "importance": imp if c["selection"] != "recency" else None, "state_k": None,
            "state_v": None, "positions": None, "cache_k": None, "cache_v": None}


def _exact_full(c, seed):
    video, n = _Video(c, seed), c["history"] * c["T"]
    past = [video.frame()[1:] for _ in range(c["history"])]
    q, k, v = video.frame()
    out = torch.zeros(q.shape, dtype=torch.float64, device=DEV)
    scores = torch.zeros((1, c["layers"], n + c["T"]), dtype=torch.float64, device=DEV)
    for l in range(c["layers"]):
        kk = torch.cat([p[0][0, l] for p in past] + [k[0, l]])
        vv = torch.cat([p[1][0, l] for p in past] + [v[0, l]])
        out[0, l], w = _attend(q[0, l], kk, vv, n)
        scores[0, l] = w.sum(dim=0)
    return {"out": out, "scores": scores} if c["scores"] else {"out": out}


def _exact_decode(c, seed):
    video, n = _Video(c, seed), c["history"] * c["T"]
    past = [video.frame()[1:] for _ in range(c["history"])]
    q, k, v = video.frame(c["tokens"])
    outs = []
    for l in range(c["layers"]):
        kk = torch.cat([p[0][0, l] for p in past] + [k[0, l]])
        vv = torch.cat([p[1][0, l] for p in past] + [v[0, l]])
        outs.append(_attend(q[0, l], kk, vv, n)[0][None, None])
    return {"out": outs, "cache_k": None, "cache_v": None}


def _exact_block(c, seed):
    bs, weights, x = _block_parts(c, seed)
    S, L, T, d, hq, hkv = c["streams"], c["layers"], c["T"], c["d"], c["hq"], c["hkv"]
    freq = bs.rope_theta ** (-2.0 * torch.arange(d // 2, device=DEV, dtype=torch.float64) / d)

    def norm(a, g):
        return a * torch.rsqrt(a.square().mean(dim=-1, keepdim=True) + bs.rms_eps) * g.double()

    def rotate(a, pos):
        ang = pos[:, None, None] * freq
        a1, a2 = a[..., : d // 2], a[..., d // 2:]
        return torch.cat([a1 * ang.cos() - a2 * ang.sin(), a2 * ang.cos() + a1 * ang.sin()], dim=-1)

    h = [f.double() for f in x[:3]]  # the first timed pass and the two frames before it
    for l in range(L):
        w = weights[l]
        wqkv, wo = w["w_qkv"].double().t(), w["w_o"].double().t()
        past = [[] for _ in range(S)]
        mid = []
        for n in range(3):
            qkv = torch.matmul(norm(h[n], w["norm_attn"]), wqkv) + w["b_qkv"].double()
            pos = n * T + torch.arange(T, device=DEV, dtype=torch.float64)
            o = torch.empty((S, T, hq * d), dtype=torch.float64, device=DEV)
            for s in range(S):
                q, k, v = (a.view(T, -1, d) for a in qkv[s].split([hq * d, hkv * d, hkv * d], dim=-1))
                past[s].append((rotate(k, pos), v))
                kk, vv = (torch.cat([p[i] for p in past[s]]) for i in (0, 1))
                o[s] = _attend(rotate(q, pos), kk, vv, n * T)[0].reshape(T, hq * d)
            mid.append(h[n] + torch.matmul(o, wo))
        del wqkv, wo
        wgu, wd = w["w_gate_up"].double().t(), w["w_down"].double().t()
        for n in range(3):
            gu = torch.matmul(norm(mid[n], w["norm_mlp"]), wgu)
            gate, up = gu.chunk(2, dim=-1)
            h[n] = mid[n] + torch.matmul(torch.nn.functional.silu(gate) * up, wd)
    return {"out": h[2], "state_k": None, "state_v": None, "positions": None, "cache_k": None,
            "cache_v": None}


def _exact_diagnose(c, seed):
    now, nxt = _diagnose_scores(c, seed)
    n, T, B = c["n_hist"], c["T"], c["B"]

    def top(s, m, b):
        keep = torch.zeros(s.shape, dtype=torch.bool, device=DEV)
        at = torch.sort(s[:, :m], dim=1, descending=True, stable=True).indices[:, : min(b, m)]
        return keep.scatter_(1, at, True)

    x, y = now.double(), nxt.double()
    conc = [(x * top(now, n, b))[:, :n].sum(1) / x[:, :n].sum(1) for b in (max(1, B // 8), B)]
    s_n, s_next = top(now, n, B), top(nxt, n + T, B)
    pool = s_n.clone()
    pool[:, n: n + T] = True
    count = s_next.sum(1).double()
    both = (s_n & s_next).sum(1).double()
    return {"mask": None, "concentration": torch.stack(conc, dim=1),
            "recall": (s_next & pool).sum(1).double() / count,
            "weighted_recall": (y * (s_next & pool)).sum(1) / (y * s_next).sum(1),
            "retention": both / s_n.sum(1).double(), "churn": (count - both) / count}
