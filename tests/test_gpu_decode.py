"""statekv_decode_step: decoding over the detailed cache (Sec. 3.2 / 3.3).

After a video has been prefilled frame by frame, text tokens (a prompt, then
one generated token per call) attend to every row of the decode cache and
causally to each other.  The output must equal the oracle's exact attention
over the video frames' K/V (taken from the input generator) followed by the
text tokens' K/V; the cache rows must be bit copies of every input; once a
(stream, layer) has decoded, prefill is refused and the cache capacity holds.
"""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2605_31598_gb300 import StateKV, make_config
from paper_2605_31598_gb300.inputs import WORKLOADS, batch_qkv

from .parity import OUT_ATOL


def _text_tokens(shape, n, seed, device):
    """Seeded synthetic text-token Q/K/V, [S][L][n][H][d] bf16, N(0,1)/sqrt(d)."""
    g = torch.Generator(device="cpu").manual_seed(seed)
    S, L, d = shape.num_streams, shape.num_layers, shape.head_dim
    mk = lambda h: (torch.randn((S, L, n, h, d), generator=g) * d ** -0.5).to(torch.bfloat16)
    return (mk(shape.num_q_heads).to(device), mk(shape.num_kv_heads).to(device),
            mk(shape.num_kv_heads).to(device))


@pytest.mark.gpu
@pytest.mark.parametrize("name,frames,steps,units", [
    ("toy", 4, (5, 1, 1, 1), [(0, 0)]),
    # end of a 12-frame video on the 28-layer stack: 2352 video rows, a 32-token
    # prompt, then two generated tokens
    ("qwen7b_stack", 12, (32, 1, 1), [(0, 0), (0, 27)]),
])
def test_decode_matches_exact_oracle(name, frames, steps, units):
    import __graft_entry__ as g

    g.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    base = WORKLOADS[name]
    T = base.tokens_per_frame
    extra = -(-sum(steps) // T)  # frames of capacity the text rows need
    shape = dataclasses.replace(base, max_frames=frames + extra)
    S, L = shape.num_streams, shape.num_layers
    eng = StateKV(make_config(shape))
    hist = {u: ([], []) for u in units}
    for n in range(1, frames + 1):
        q, k, v = batch_qkv(shape, n, streams=range(S), layers=range(L), device="cuda")
        for u in units:
            hist[u][0].append(oracle.as_bf16_bits(k[u]))
            hist[u][1].append(oracle.as_bf16_bits(v[u]))
        assert eng.prefill_frame(q, k, v, torch.empty_like(q)) == 0
    done = frames * T
    for i, nt in enumerate(steps):
        q, k, v = _text_tokens(shape, nt, seed=100 + i, device="cuda")
        out = torch.full_like(q, float("nan"))
        assert eng.decode_step(q, k, v, out) == 0
        torch.cuda.synchronize()
        for u in units:
            ks = np.concatenate(hist[u][0] + [oracle.as_bf16_bits(k[u])])
            vs = np.concatenate(hist[u][1] + [oracle.as_bf16_bits(v[u])])
            ref = oracle.full_attention(oracle.as_bf16_bits(q[u]), ks, vs, done, causal=True)
            got = out[u].float().cpu().numpy()
            assert np.isfinite(got).all()
            err = float(np.abs(got - ref).max())
            assert err <= OUT_ATOL, f"step {i} ({nt} tokens) unit {u}: max |O - O_exact| = {err}"
            hist[u][0].append(oracle.as_bf16_bits(k[u]))
            hist[u][1].append(oracle.as_bf16_bits(v[u]))
        done += nt
    # the cache holds every row, bit for bit, and reports its length
    for u in units:
        ck, cv, info = eng.cache(*u)
        assert info.length == done
        assert np.array_equal(oracle.as_bf16_bits(ck[:, :done].transpose(0, 1)),
                              np.concatenate(hist[u][0]))
        assert np.array_equal(oracle.as_bf16_bits(cv[:, :done].transpose(0, 1)),
                              np.concatenate(hist[u][1]))
    # the video part is closed once a (stream, layer) has decoded
    q, k, v = batch_qkv(shape, frames + 1, streams=range(S), layers=range(L), device="cuda")
    assert eng.prefill_frame(q, k, v, torch.empty_like(q)) == 1  # INVALID_ARG
    assert eng.sync() == 0


@pytest.mark.gpu
def test_decode_refuses_rows_beyond_the_cache():
    import __graft_entry__ as g

    g.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    shape = dataclasses.replace(WORKLOADS["toy"], max_frames=3)  # 48 rows
    S, L, T = shape.num_streams, shape.num_layers, shape.tokens_per_frame
    eng = StateKV(make_config(shape))
    for n in range(1, 3):
        q, k, v = batch_qkv(shape, n, streams=range(S), layers=range(L), device="cuda")
        assert eng.prefill_frame(q, k, v, torch.empty_like(q)) == 0
    q, k, v = _text_tokens(shape, T + 1, seed=7, device="cuda")  # 32 + 17 > 48
    assert eng.decode_step(q, k, v, torch.empty_like(q)) == 3  # CACHE_FULL
    q, k, v = _text_tokens(shape, T, seed=8, device="cuda")     # exactly fills it
    assert eng.decode_step(q, k, v, torch.empty_like(q)) == 0
    q, k, v = _text_tokens(shape, 1, seed=9, device="cuda")
    assert eng.decode_step(q, k, v, torch.empty_like(q)) == 3
    assert eng.sync() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("hq,hkv,d,T,frames,layers,steps", [
    # one head: the new tokens' rows straddle a chunk's end (rows 254..257), then start one
    (4, 1, 128, 127, 2, 1, (4, 1, 3)),
    (16, 1, 64, 128, 1, 2, (1, 1)),      # 16 rows per token; the new row opens a chunk
    (2, 2, 64, 33, 1, 1, (8, 2)),        # fewer keys than a chunk
    (14, 2, 64, 259, 7, 3, (1, 2, 1)),   # ragged lengths, several units
    (7, 1, 128, 1024, 9, 1, (1, 1)),     # one head over all of its chunks (64)
])
def test_decode_token_edges(hq, hkv, d, T, frames, layers, steps):
    """One-launch decode steps (at most 16 query rows per KV head), per layer
    and over all layers in turn, against the oracle's exact attention."""
    import __graft_entry__ as g

    from paper_2605_31598_gb300.inputs import Shape

    g.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    shape = Shape(hq, hkv, d, T, 64, frames + 1, num_layers=layers, kind="peaked")
    eng = StateKV(make_config(shape))
    hist = [([], []) for _ in range(layers)]
    for n in range(1, frames + 1):
        q, k, v = batch_qkv(shape, n, streams=[0], layers=range(layers), device="cuda")
        assert eng.prefill_frame(q, k, v, torch.empty_like(q)) == 0
        for l in range(layers):
            hist[l][0].append(oracle.as_bf16_bits(k[0, l]))
            hist[l][1].append(oracle.as_bf16_bits(v[0, l]))
    done = frames * T
    for i, nt in enumerate(steps):
        q, k, v = (x * d ** 0.5 for x in _text_tokens(shape, nt, seed=300 + i, device="cuda"))
        out = torch.full_like(q, float("nan"))
        if i % 2:  # every layer in one call, else one call per layer
            assert eng.decode_step(q, k, v, out) == 0
        else:
            for l in range(layers):
                part = tuple(x[:, l:l + 1].contiguous() for x in (q, k, v, out))
                assert eng.decode_step(*part, layer_begin=l, layer_count=1) == 0
                out[:, l:l + 1] = part[3]
        torch.cuda.synchronize()
        for l in range(layers):
            hist[l][0].append(oracle.as_bf16_bits(k[0, l]))
            hist[l][1].append(oracle.as_bf16_bits(v[0, l]))
            ks, vs = np.concatenate(hist[l][0]), np.concatenate(hist[l][1])
            ref = oracle.full_attention(oracle.as_bf16_bits(q[0, l]), ks, vs, done, causal=True)
            got = out[0, l].float().cpu().numpy()
            assert np.isfinite(got).all()
            err = float(np.abs(got - ref).max())
            assert err <= OUT_ATOL, f"step {i} ({nt} tokens) layer {l}: max |O - O_exact| = {err}"
            ck, cv, info = eng.cache(0, l)
            assert info.length == done + nt
            assert np.array_equal(oracle.as_bf16_bits(ck[:, :done + nt].transpose(0, 1)), ks)
            assert np.array_equal(oracle.as_bf16_bits(cv[:, :done + nt].transpose(0, 1)), vs)
        done += nt
    assert eng.sync() == 0


@pytest.mark.gpu
@pytest.mark.parametrize("hq,d,T,frames,steps", [
    (16, 128, 1020, 8, (1, 1)),  # 16 rows over 64 chunks: merged 23 at a time, in three rounds
    (16, 64, 1020, 8, (1,)),     # 22 at a time
    (8, 128, 1020, 8, (2,)),     # two tokens of eight heads
    (16, 128, 700, 8, (1,)),     # 44 chunks, two rounds
])
def test_decode_merges_in_several_rounds(hq, d, T, frames, steps):
    """One head of 16 query rows over more chunks than the staging memory holds at once."""
    test_decode_token_edges(hq, 1, d, T, frames, 1, steps)
