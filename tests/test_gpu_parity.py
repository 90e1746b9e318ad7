"""Parity of the CUDA path (through the C ABI) with the CPU oracle on GB300.

Every case is teacher-forced (see tests/parity.py): the oracle starts each
checked frame from the GPU's pre-frame state and the outputs, importance,
selection, state rows and decode cache are compared.
"""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2605_31598_gb300 import StateKV, make_config
from paper_2605_31598_gb300.inputs import WORKLOADS, Shape, batch_qkv

from .parity import IMP_ATOL, IMP_RTOL, OUT_ATOL, run_free_running, run_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g

    g.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_smoke():
    import __graft_entry__ as g

    g.smoke()


def test_toy_all_frames():
    """The toy layer (d 64, T 16, B 32, 8 frames): every frame checked."""
    stats = {}
    run_parity(WORKLOADS["toy"], 8, stats=stats)
    print("toy", stats)


def test_qwen7b_layer_sampled_frames():
    """One Qwen2-7B-shaped layer (28q/4kv, d 128, T 196, B 1568), 64 frames:
    fill, first eviction and late frames checked."""
    stats = {}
    run_parity(WORKLOADS["qwen7b_layer"], 64, check_frames=[1, 2, 8, 9, 10, 11, 33, 64],
               stats=stats)
    print("qwen7b_layer", stats)


def test_peaked_inputs_selection():
    """Unit-variance Q/K (far from uniform attention): many frame tokens win
    slots each frame, so the selection is exercised well outside the band."""
    shape = dataclasses.replace(WORKLOADS["qwen7b_layer"], max_frames=16)
    stats = {}
    run_parity(shape, 14, kind="peaked", check_frames=[9, 10, 11, 12, 14], stats=stats)
    print("peaked", stats)
    assert stats["decisions"] > 0


EDGE = {
    "g1_d64": Shape(2, 2, 64, 50, 80, 6),
    "g8_d128_t33": Shape(16, 2, 128, 33, 40, 5),
    "b_lt_t": Shape(7, 1, 128, 196, 50, 4),
    "b0": Shape(4, 2, 64, 40, 0, 3),
    "t300_three_frame_tiles": Shape(4, 1, 128, 300, 256, 4),
    "t1": Shape(4, 2, 64, 1, 3, 6),
    "tile_multiples": Shape(2, 1, 128, 128, 256, 5),
    "g7_d64": Shape(7, 1, 64, 20, 24, 5),
}


@pytest.mark.parametrize("name", sorted(EDGE))
def test_edge_shapes(name):
    shape = EDGE[name]
    run_parity(shape, shape.max_frames, kind="peaked")


def test_bidirectional_in_frame_variant():
    run_parity(WORKLOADS["toy"], 5, causal=False)


def test_multi_stream_multi_layer_split_calls():
    """Two streams x three layers, each frame issued as two calls over layer
    ranges [0, 2) and [2, 3)."""
    shape = Shape(8, 2, 128, 64, 96, 5, num_layers=3, num_streams=2)
    run_parity(shape, 5, call_layers=[(0, 2), (2, 1)])


def test_without_importance_export():
    run_parity(WORKLOADS["toy"], 4, want_importance=False)


def test_host_buffer_entry_point():
    run_parity(Shape(8, 2, 128, 64, 96, 4, num_layers=2), 4, host_api=True)


def test_pipelined_host_frames_match_device_calls():
    """statekv_prefill_frames_host (copies on internal streams, two staging
    sets) leaves outputs, importance and states bit-identical to one
    statekv_prefill_frame per frame: two pipelined calls in a row, then a
    single-frame host call that reuses the first staging set."""
    shape = Shape(8, 2, 128, 64, 96, 8, num_layers=2, num_streams=2)
    S, L, H, P = 2, 2, 2, 96 + 64
    dev = StateKV(make_config(shape))
    hst = StateKV(make_config(shape, host_staging=True))
    frames = [batch_qkv(shape, n, streams=range(S), layers=range(L), device="cuda")
              for n in range(1, 8)]
    want = []
    for q, k, v in frames:
        o = torch.empty_like(q)
        imp = torch.empty((S, L, H, P), dtype=torch.float32, device="cuda")
        assert dev.prefill_frame(q, k, v, o, imp) == 0
        want.append((o, imp))
    host = [tuple(x.cpu().pin_memory() for x in (q, k, v)) +
            (torch.empty(q.shape, dtype=torch.bfloat16).pin_memory(),
             torch.empty((S, L, H, P), dtype=torch.float32).pin_memory())
            for q, k, v in frames]
    # refused before any work: mixed importance buffers, too many frames
    mixed = [host[0], host[1][:4] + (None,)]
    assert hst.prefill_frames_host(mixed) == 1
    assert hst.prefill_frames_host(host * 2) == 3  # 14 frames > max_frames = 8
    torch.cuda.synchronize()
    assert hst.state(0, 0)[3].frames == 0
    assert hst.prefill_frames_host(host[:3]) == 0
    assert hst.prefill_frames_host(host[3:6]) == 0
    assert hst.prefill_frame_host(*host[6]) == 0
    torch.cuda.synchronize()
    for n, (o, imp) in enumerate(want):
        assert torch.equal(host[n][3].view(torch.int16), o.cpu().view(torch.int16)), f"out, frame {n + 1}"
        assert torch.equal(host[n][4], imp.cpu()), f"importance, frame {n + 1}"
    for s_ in range(S):
        for l_ in range(L):
            a, b = dev.state(s_, l_), hst.state(s_, l_)
            assert a[3].frames == b[3].frames == 7 and a[3].count == b[3].count
            for x, y in zip(a[:3], b[:3]):
                assert torch.equal(x.view(torch.int16) if x.dtype == torch.bfloat16 else x,
                                   y.view(torch.int16) if y.dtype == torch.bfloat16 else y)
    assert dev.sync() == 0 and hst.sync() == 0


def test_cache_full_is_refused_without_side_effects():
    shape = Shape(4, 1, 64, 16, 32, 2)
    eng = StateKV(make_config(shape))
    for n in (1, 2):
        q, k, v = batch_qkv(shape, n, streams=[0], layers=[0], device="cuda")
        assert eng.prefill_frame(q, k, v, torch.empty_like(q)) == 0
    torch.cuda.synchronize()
    kk, vv, pp, info = eng.state(0, 0)
    before = (kk.clone(), pp.clone(), info.frames)
    q, k, v = batch_qkv(shape, 3, streams=[0], layers=[0], device="cuda")
    assert eng.prefill_frame(q, k, v, torch.empty_like(q)) == 3  # CACHE_FULL
    torch.cuda.synchronize()
    kk, vv, pp, info = eng.state(0, 0)
    assert torch.equal(kk, before[0]) and torch.equal(pp, before[1]) and info.frames == 2
    assert eng.sync() == 0


def test_invalid_ranges_and_alignment_enqueue_nothing():
    shape = Shape(4, 1, 64, 16, 32, 4, num_layers=2)
    eng = StateKV(make_config(shape))
    q, k, v = batch_qkv(shape, 1, streams=[0], layers=[0, 1], device="cuda")
    out = torch.empty_like(q)
    assert eng.prefill_frame(q, k, v, out, layer_begin=1, layer_count=2) == 1
    assert eng.prefill_frame(q, k, v, out, stream_begin=1, stream_count=1) == 1
    flat = torch.empty(q.numel() + 8, dtype=torch.bfloat16, device="cuda")
    qmis = flat[1:1 + q.numel()].view_as(q)  # 2-byte offset: not 16-byte aligned
    assert eng.prefill_frame(qmis, k, v, out) == 1
    torch.cuda.synchronize()
    assert eng.state(0, 0)[3].frames == 0


def test_determinism_bit_identical():
    shape = Shape(28, 4, 128, 196, 1568, 12)
    outs = []
    for _ in range(2):
        eng = StateKV(make_config(shape))
        res = []
        for n in range(1, 12):
            q, k, v = batch_qkv(shape, n, streams=[0], layers=[0], device="cuda")
            out = torch.empty_like(q)
            imp = torch.empty((1, 1, 4, shape.state_capacity + 196), device="cuda")
            assert eng.prefill_frame(q, k, v, out, imp) == 0
            res.append((out.clone(), imp.clone()))
        kk, vv, pp, _ = eng.state(0, 0)
        torch.cuda.synchronize()
        outs.append((res, kk.clone(), pp.clone()))
        eng.close()
    for (a, b) in zip(outs[0][0], outs[1][0]):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert torch.equal(outs[0][1], outs[1][1]) and torch.equal(outs[0][2], outs[1][2])


def test_qwen7b_stack_full_size_sampled_units():
    """The 28-layer 7B stack at full size (B 2048), in the one-call-per-frame
    launch configuration the benchmark times: frame 12 (first frames after
    the state fills) compared in full on two of the 28 layers."""
    shape = WORKLOADS["qwen7b_stack"]
    stats = {}
    run_parity(shape, 12, check_frames=[11, 12], units=[(0, 0), (0, 27)], stats=stats)
    print("qwen7b_stack", stats)


def test_qwen7b_stack_late_frames():
    """The 28-layer 7B stack carried to frame 256, the last frame of its
    workload (positions up to 50,175; 245 frames of state churn after the
    state fills), in the benchmark's one-call-per-frame launch: frames 128
    and 256 compared in full on three of the 28 layers."""
    stats = {}
    run_parity(WORKLOADS["qwen7b_stack"], 256, check_frames=[128, 256],
               units=[(0, 0), (0, 13), (0, 27)], stats=stats)
    print("qwen7b_stack late", stats)


def test_qwen72b_stack_first_evictions():
    """The 80-layer 72B-shaped stack (64 q / 8 kv heads, B 4096: 33 state key
    tiles per unit, a 4292-member pool) in its one-launch-per-frame
    configuration: frame 21 (the first whose pool exceeds B) and frame 24
    compared in full on three of the 80 layers.  The decode cache is sized
    for 24 frames; the launch does not depend on it."""
    shape = dataclasses.replace(WORKLOADS["qwen72b_stack"], max_frames=24)
    stats = {}
    run_parity(shape, 24, check_frames=[21, 24], units=[(0, 0), (0, 41), (0, 79)], stats=stats)
    print("qwen72b_stack", stats)


def test_qwen7b_8streams_late_frame():
    """Eight concurrent 7B streams (28 layers each, 224 units per launch)
    carried to frame 1024, the end of the streaming workload (virtual
    positions up to 200,703): frames 512 and 1024 compared in full on one
    layer of each of two streams."""
    stats = {}
    run_parity(WORKLOADS["qwen7b_8streams"], 1024, check_frames=[512, 1024],
               units=[(2, 5), (6, 27)], stats=stats)
    print("qwen7b_8streams late", stats)


FREE_RUNNING = {
    # the toy layer over 32 frames: its first near-tie comes at frame 13
    "toy": (dataclasses.replace(WORKLOADS["toy"], max_frames=32), None),
    # one KV head of 4 query heads, d 128, T 64, B 128, unit-variance Q/K:
    # first near-tie at frame 8
    "peaked_g4_t64": (Shape(4, 1, 128, 64, 128, 32), "peaked"),
}


@pytest.mark.parametrize("name", sorted(FREE_RUNNING))
def test_free_running_until_first_near_tie(name):
    """The GPU and the oracle each keep their own state from frame 1 (no
    teacher forcing): the kept position sets must agree after every frame
    until the first frame whose selection boundary is a near-tie."""
    shape, kind = FREE_RUNNING[name]
    stats = {}
    n, tie = run_free_running(shape, shape.max_frames, kind=kind, stats=stats)
    print("free running", name, stats)
    first_eviction = shape.state_capacity // shape.tokens_per_frame + 1
    assert n >= first_eviction + 2  # several evicting frames matched exactly


@pytest.mark.gpu
def test_streams_at_different_frames_in_one_launch():
    """One launch whose units see different key ranges: stream 0 runs three
    frames ahead of stream 1, so the persistent attention kernel walks units
    with different state sizes (and tile counts) side by side.  Every frame
    of both streams is checked against the oracle started from the GPU's
    pre-frame state (outputs within 2e-2, importance within 1e-3)."""
    import numpy as np

    import oracle
    from paper_2605_31598_gb300 import StateKV, make_config
    from paper_2605_31598_gb300.inputs import batch_qkv

    from .parity import IMP_ATOL, IMP_RTOL, OUT_ATOL

    shape = Shape(8, 2, 128, 64, 160, 9, num_layers=2, num_streams=2)
    S, L, T, Hq, Hkv, d, B = 2, 2, 64, 8, 2, 128, 160
    eng = StateKV(make_config(shape))
    lays = {(s, l): oracle.OracleLayer(Hq, Hkv, d, T, B, shape.max_frames) for s in range(S) for l in range(L)}
    done = [0, 0]

    def run(streams):
        frames = [done[s] + 1 for s in streams]
        q, k, v = batch_qkv(shape, frames, streams=streams, layers=range(L), device="cuda")
        torch.cuda.synchronize()
        pre = {}
        for si, s in enumerate(streams):
            for l in range(L):
                kk, vv, pp, info = eng.state(s, l)
                pre[(s, l)] = (info.count, pp.cpu().numpy().astype(np.int64), oracle.as_bf16_bits(kk),
                               oracle.as_bf16_bits(vv), info.virtual_len)
        out = torch.full_like(q, float("nan"))
        imp = torch.full((len(streams), L, Hkv, B + T), float("nan"), device="cuda")
        assert eng.prefill_frame(q, k, v, out, imp, stream_begin=streams[0],
                                 stream_count=len(streams)) == 0
        torch.cuda.synchronize()
        for si, s in enumerate(streams):
            for l in range(L):
                count, ppos, pk, pv, vlen = pre[(s, l)]
                lay = lays[(s, l)]
                lay.set_state(np.full(Hkv, count, np.int32), ppos, pk, pv, vlen)
                o_ref, imp_ref, _ = lay.prefill_frame(*(oracle.as_bf16_bits(x[si, l]) for x in (q, k, v)))
                err = float(np.abs(out[si, l].float().cpu().numpy() - o_ref).max())
                assert err <= OUT_ATOL, (s, l, done[s] + 1, err)
                g = imp[si, l].cpu().numpy().astype(np.float64)
                for h in range(Hkv):
                    order = {int(p): i for i, p in enumerate(np.sort(ppos[h, :count]))}
                    ref = np.array([imp_ref[h, order[int(ppos[h, j])]] for j in range(count)] +
                                   list(imp_ref[h, B:]))
                    got = np.concatenate([g[h, :count], g[h, B:]])
                    assert np.all(np.abs(got - ref) <= IMP_RTOL * np.abs(ref) + IMP_ATOL), (s, l, h)
        for s in streams:
            done[s] += 1

    for _ in range(3):
        run([0])
    for _ in range(5):
        run([0, 1])
    assert done == [8, 5]
    assert eng.sync() == 0


# few work units over many key tiles: the attention kernel's split form (a cluster
# of CTAs per unit), from two CTAs to eight, with ragged last tiles
SPLIT = {
    "one_unit_d128": (Shape(2, 1, 128, 64, 1100, 22), 22),
    "three_units_ragged_d64": (Shape(6, 3, 64, 37, 700, 24), 24),
    "long_frame_b0_like": (Shape(1, 1, 128, 300, 2500, 10), 10),
    "frame_tiles_only": (Shape(1, 1, 64, 900, 0, 2), 2),
}


@pytest.mark.parametrize("name", sorted(SPLIT))
@pytest.mark.parametrize("causal", [True, False])
def test_split_attention_parity(name, causal):
    shape, frames = SPLIT[name]
    run_parity(shape, frames, kind="peaked", causal=causal,
               check_frames=[f for f in (1, 2, frames // 2, frames) if f <= frames])


def test_split_attention_with_streams_at_different_frames():
    """A stream that has seen 16 frames and one at its first share a call: the
    CTAs per unit follow the longer one, so some of the other's CTAs hold no key
    tile.  The short stream's outputs equal those of a call of its own."""
    shape = Shape(4, 1, 128, 64, 1000, 20, num_streams=2, kind="peaked")
    B, T = shape.state_capacity, shape.tokens_per_frame
    both, own = StateKV(make_config(shape)), StateKV(make_config(shape))
    for n in range(1, 17):
        q, k, v = batch_qkv(shape, n, streams=[0], layers=[0], device="cuda")
        assert both.prefill_frame(q, k, v, torch.empty_like(q), stream_begin=0, stream_count=1) == 0
    q, k, v = batch_qkv(shape, [17, 1], streams=[0, 1], layers=[0], device="cuda")
    out, imp = torch.full_like(q, float("nan")), torch.full((2, 1, 1, B + T), float("nan"), device="cuda")
    assert both.prefill_frame(q, k, v, out, imp) == 0
    out1, imp1 = torch.empty_like(q[1:]), torch.empty((1, 1, 1, B + T), device="cuda")
    assert own.prefill_frame(q[1:].contiguous(), k[1:].contiguous(), v[1:].contiguous(), out1, imp1,
                             stream_begin=1, stream_count=1) == 0
    torch.cuda.synchronize()
    assert both.sync() == 0 and own.sync() == 0
    assert torch.isfinite(out).all() and torch.isfinite(imp).all()
    assert (out[1:].float() - out1.float()).abs().max().item() <= OUT_ATOL
    torch.testing.assert_close(imp[1:], imp1, rtol=IMP_RTOL, atol=IMP_ATOL)


SELECT = {
    # (shape, zero queries: importance ties by the hundred, frames)
    "one_pass": (Shape(4, 2, 64, 16, 64, 8, num_layers=3, num_streams=2), False, 8),
    "ties": (Shape(2, 2, 64, 48, 1500, 36), True, 36),
    "ties_member_wise": (Shape(2, 1, 64, 33, 700, 25, num_layers=2), True, 25),
    "large_member_wise": (Shape(2, 1, 128, 50, 3001, 62), False, 62),
    "large_ties": (Shape(2, 2, 64, 100, 6000, 62), True, 62),
    "large": (Shape(2, 2, 64, 200, 11000, 57, num_layers=2), False, 57),
    "many_heads": (Shape(16, 16, 64, 100, 6000, 62), False, 62),
    "eight_ctas": (Shape(2, 2, 64, 400, 21600, 57), False, 57),
    "eight_ctas_member_wise": (Shape(2, 1, 64, 401, 11000, 30), False, 30),
}


@pytest.mark.parametrize("selection", [0, 2])
@pytest.mark.parametrize("name", sorted(SELECT))
def test_selection_is_exact_for_the_exported_importance(name, selection):
    """The kept positions, slot by slot: the B pool members largest in (importance,
    earlier position), freed slots in ascending order taken by the admitted tokens
    in ascending order.  The ranking is redone from the importance the step exports
    (layer mode: summed over the heads in order, in fp32), so nothing is rounded."""
    shape, zero_q, frames = SELECT[name]
    S, L, H, T, B = (shape.num_streams, shape.num_layers, shape.num_kv_heads, shape.tokens_per_frame,
                     shape.state_capacity)
    eng = StateKV(make_config(shape, selection=selection))
    for n in range(1, frames + 1):
        q, k, v = batch_qkv(shape, n, streams=list(range(S)), layers=list(range(L)), device="cuda")
        if zero_q:
            q = torch.zeros_like(q)
        imp = torch.full((S, L, H, B + T), float("nan"), device="cuda")
        if n > frames - 3:
            torch.cuda.synchronize()
            before = [[eng.state(s, l)[2].cpu().numpy().copy() for l in range(L)] for s in range(S)]
        assert eng.prefill_frame(q, k, v, torch.empty_like(q), imp) == 0
        if n <= frames - 3:
            continue
        torch.cuda.synchronize()
        count = min(B, (n - 1) * T)
        imps = imp.cpu().numpy()
        for s in range(S):
            for l in range(L):
                after = eng.state(s, l)[2].cpu().numpy()
                for h in range(H):
                    x = imps[s, l, h]
                    if selection == 2:
                        x = np.zeros(B + T, np.float32)
                        for h2 in range(H):
                            x = x + imps[s, l, h2]
                    pos = np.concatenate([before[s][l][h][:count], (n - 1) * T + np.arange(T)]).astype(np.int64)
                    sc = np.concatenate([x[:count], x[B:]])
                    kept = np.zeros(count + T, bool)
                    kept[np.lexsort((pos, -sc))[:B]] = True
                    want = np.full(B, -1, np.int64)
                    want[:count] = pos[:count]
                    free = [i for i in range(B) if i >= count or not kept[i]]
                    adm = [t for t in range(T) if kept[count + t]]
                    for i, t in zip(free, adm):
                        want[i] = (n - 1) * T + t
                    live = min(B, count + T)
                    got = after[h].astype(np.int64)
                    assert (got[:live] == want[:live]).all(), (name, n, s, l, h)
    assert eng.sync() == 0


FEW_TILES = {
    # (shape, frames): 64 heads (a CTA each) whose pools are taken member by member.  With
    # at most four query tiles and a pool above 2560 the sums are formed eight members at a
    # time, else two at a time.
    "one_tile_two_rounds": (Shape(32, 32, 64, 100, 5201, 55, num_layers=2), 55),
    "four_tiles": (Shape(32, 8, 64, 128, 2501, 22, num_layers=8), 22),
    "five_tiles": (Shape(32, 8, 64, 129, 2502, 22, num_layers=8), 22),
    "pool_2557": (Shape(32, 32, 64, 100, 2457, 27, num_layers=2), 27),
    "pool_2561": (Shape(32, 32, 64, 100, 2461, 27, num_layers=2), 27),
}


@pytest.mark.parametrize("name", sorted(FEW_TILES))
def test_layer_selection_is_exact_with_few_query_tiles(name, monkeypatch):
    """As above, for layer-level scores over few query tiles."""
    shape, frames = FEW_TILES[name]
    monkeypatch.setitem(SELECT, name, (shape, False, frames))
    test_selection_is_exact_for_the_exported_importance(name, 2)


def test_append_with_64_bit_indexes():
    """One frame of 4096 tokens of 16,384 KV heads of 128 (2^31 copies of 16 bytes): every
    row is in the decode cache.  About 95 GB on the device."""
    if torch.cuda.mem_get_info()[0] < 120e9:
        pytest.skip("needs 120 GB of free device memory")
    H, T, d = 16384, 4096, 128
    eng = StateKV(make_config(Shape(H, H, d, T, 0, 1)))
    g = torch.Generator(device="cuda")
    g.manual_seed(0)
    k, v = (torch.empty((1, 1, T, H, d), dtype=torch.bfloat16, device="cuda").normal_(generator=g) for _ in range(2))
    out = torch.empty_like(k)
    assert eng.prefill_frame(k, k, v, out) == 0
    assert eng.sync() == 0
    ck, cv, info = eng.cache(0, 0)
    assert info.length == T
    for h in range(0, H, 2048):
        for rows, src in ((ck, k), (cv, v)):
            assert torch.equal(rows[h:h + 2048], src[0, 0, :, h:h + 2048].transpose(0, 1)), h
    eng.close()
    del eng, k, v, out, ck, cv
    torch.cuda.empty_cache()
