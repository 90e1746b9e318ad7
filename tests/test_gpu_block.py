"""The full per-frame transformer block (statekv_block_frame) against the
block oracle, teacher-forced layer by layer: each layer runs on the GPU alone
(layer_count = 1), and the oracle layer starts from the GPU's input hidden
states and the GPU's pre-frame StateKV state of that layer.

Tolerance of the layer output x2 (bf16 [T][hidden]): the attention output may
differ by up to 2e-2 (the step's bound), which the output projection maps to
about sqrt(Hq d) * std(W_o) times that on each x1 entry; bf16 rounding of
intermediates adds a few ulps (2^-8 relative each), and GPU (fp32) and oracle
(fp64) sums sometimes round to neighbouring bf16 values.  The test asserts
|dx| <= 2^-6 |x| + 3 * 2e-2 * sqrt(Hq d) * std(W_o) per entry, and an RMS
error within half a bf16 ulp of the RMS value (2^-7 relative) plus a tenth
of the attention term.  Selections agree outside the 1e-3 band
of the oracle's importance, and the decode caches hold the GPU's own
rotated K/V rows bit for bit.
"""
import ctypes
import dataclasses
import math

import numpy as np
import pytest
import torch

import oracle
from oracle import block as ob
from paper_2605_31598_gb300 import StateKV, make_config, statekv
from paper_2605_31598_gb300.inputs import (BLOCKS, WORKLOADS, Shape, block_input,
                                           block_weights)
from paper_2605_31598_gb300.statekv import block_weights_array, statekv_block_config

from .parity import BAND

F64 = lambda t: t.double().cpu().numpy()


def _need_gpu():
    import __graft_entry__ as g

    g.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _oracle_weights(w):
    return ob.BlockWeights(F64(w["norm_attn"]), F64(w["w_qkv"]),
                           F64(w["b_qkv"]) if w["b_qkv"] is not None else None, F64(w["w_o"]),
                           F64(w["norm_mlp"]), F64(w["w_gate_up"]), F64(w["w_down"]))


def run_block_parity(shape, block, nframes, *, check_frames=None, yarn=(1.0, 0), bias=True,
                     stats=None):
    S, L = shape.num_streams, shape.num_layers
    T, Hq, Hkv, d, B = (shape.tokens_per_frame, shape.num_q_heads, shape.num_kv_heads,
                        shape.head_dim, shape.state_capacity)
    eng = StateKV(make_config(shape))
    bc = statekv_block_config(block.hidden, block.intermediate, block.rms_eps, block.rope_theta,
                              yarn[0], yarn[1])
    wts = block_weights(shape, block, device="cuda", bias=bias)
    warr = block_weights_array(wts)
    ws = torch.empty(eng.block_workspace_bytes(bc), dtype=torch.uint8, device="cuda")
    ows = [_oracle_weights(w) for w in wts]
    blocks = [ob.OracleBlock(Hq, Hkv, d, T, B, shape.max_frames, ows, eps=block.rms_eps,
                             theta=block.rope_theta, yarn_factor=yarn[0], original_max=yarn[1])
              for _ in range(S)]
    bound_abs = 3 * 2e-2 * math.sqrt(Hq * d) * block.weight_std
    worst = 0.0
    stats = stats if stats is not None else {}
    check_frames = set(range(1, nframes + 1) if check_frames is None else check_frames)
    for n in range(1, nframes + 1):
        x = block_input(shape, block, n, device="cuda")
        for l in range(L):
            checking = n in check_frames
            pre = []
            if checking:
                torch.cuda.synchronize()
                for s in range(S):
                    kk, vv, pp, info = eng.state(s, l)
                    pre.append((info.count, pp.cpu().numpy().astype(np.int64),
                                oracle.as_bf16_bits(kk), oracle.as_bf16_bits(vv),
                                info.virtual_len))
            y = torch.empty_like(x)
            rc = eng.block_frame(bc, warr, x, y, ws, layer_begin=l, layer_count=1)
            assert rc == 0, f"frame {n} layer {l}: statekv_block_frame returned {rc}"
            if checking:
                torch.cuda.synchronize()
                for s in range(S):
                    count, ppos, pk, pv, vlen = pre[s]
                    lay = blocks[s].layers[l]
                    lay.set_state(np.full(Hkv, count, np.int32), ppos, pk, pv, vlen)
                    ref, mid = blocks[s].layer_frame(l, F64(x[s]))
                    g = F64(y[s])
                    err = np.abs(g - ref)
                    worst = max(worst, float(err.max()))
                    ok = err <= 2 ** -6 * np.abs(ref) + bound_abs
                    assert ok.all(), (f"frame {n} layer {l} stream {s}: worst |dx| {err.max()}"
                                      f" (bound {bound_abs})")
                    rms_err = math.sqrt(np.mean(err ** 2))
                    rms_ref = math.sqrt(np.mean(ref ** 2))
                    stats["rms_rel"] = max(stats.get("rms_rel", 0.0), rms_err / rms_ref)
                    assert rms_err <= 2 ** -7 * rms_ref + bound_abs / 10, (rms_err, rms_ref)
                    # selection outside the band of the oracle's importance
                    kk, vv, pp, info = eng.state(s, l)
                    post = pp.cpu().numpy()
                    imp, kept = mid["imp"], mid["kept"]
                    for h in range(Hkv):
                        gset = set(int(p) for p in post[h] if p >= 0)
                        assert len(gset) == min(B, count + T)
                        cand_pos = np.concatenate([np.sort(ppos[h, :count]), vlen + np.arange(T)])
                        cand = np.concatenate([imp[h, :count], imp[h, B:]])
                        ck = np.concatenate([kept[h, :count], kept[h, B:]]).astype(bool)
                        if count + T > B and B > 0:
                            tau = np.sort(cand)[::-1][B - 1]
                            outside = np.abs(cand - tau) > BAND * tau
                        else:
                            outside = np.ones(len(cand), bool)
                        gk = np.array([int(p) in gset for p in cand_pos])
                        assert not (outside & (gk != ck)).any(), f"frame {n} layer {l}: selection"
                    # the decode cache's new rows are the GPU's rotated K: equal to the
                    # oracle's except where a projection sum rounded to a neighbouring
                    # bf16 value (one input ulp, up to 2^-6 at |k| < 4, moves a rotated
                    # entry by about as much)
                    ck_, cv_, cinfo = eng.cache(s, l)
                    assert cinfo.length == n * T
                    k_new = F64(ck_[:, (n - 1) * T: n * T].transpose(0, 1))
                    np.testing.assert_allclose(k_new, mid["k"], rtol=2 ** -6, atol=2 ** -6)
                    assert np.mean(k_new == mid["k"]) > 0.95
            x = y
    assert eng.sync() == 0
    return worst


@pytest.mark.gpu
def test_block_tiny_two_layers_two_streams_with_eviction():
    _need_gpu()
    shape = Shape(4, 2, 64, 16, 32, 6, num_layers=2, num_streams=2)
    stats = {}
    worst = run_block_parity(shape, BLOCKS["tiny"], 6, stats=stats)
    print("tiny block worst |dx|", worst, stats)


@pytest.mark.gpu
def test_block_tiny_yarn_scaled_rope_without_bias():
    _need_gpu()
    shape = Shape(2, 1, 128, 16, 24, 4, num_layers=2)
    run_block_parity(shape, BLOCKS["tiny"], 4, yarn=(4.0, 32), bias=False)


@pytest.mark.gpu
def test_block_qwen7b_geometry_two_layers():
    """The 7B layer widths (hidden 3584, MLP 18944, 28/4 heads, d 128), two
    layers, three frames of one stream."""
    _need_gpu()
    shape = dataclasses.replace(WORKLOADS["qwen7b_layer"], num_layers=2, max_frames=3)
    stats = {}
    worst = run_block_parity(shape, BLOCKS["qwen7b"], 3, check_frames=[1, 3], stats=stats)
    print("7B block worst |dx|", worst, stats)


@pytest.mark.gpu
def test_block_ragged_widths_many_streams():
    """Widths that are not multiples of the GEMM tiles (hidden 136, MLP 200:
    ragged 128-column tiles and a ragged last 64-wide K step) and 20 streams
    (320 rows: two 256-row pairs, the second only partly filled), so the
    projections take several row pairs and split K."""
    from paper_2605_31598_gb300.inputs import BlockShape

    _need_gpu()
    shape = Shape(4, 2, 64, 16, 32, 3, num_layers=1, num_streams=20)
    stats = {}
    worst = run_block_parity(shape, BlockShape(136, 200, weight_std=0.08), 3, stats=stats)
    print("ragged block worst |dx|", worst, stats)


@pytest.mark.gpu
def test_block_ragged_widths_thin_rows():
    """At most 256 rows (here 4 streams x 49 tokens = 196, one stream's row
    count at 7B shape) the projections run as thin GEMMs writing split-K
    partials that the RoPE, residual and SiLU kernels add up.  Hidden 136 and
    MLP 200 give ragged W row blocks, a ragged last K step, and a gate/up
    projection with only two row-block pairs, so it splits K and its SiLU
    reads partials."""
    from paper_2605_31598_gb300.inputs import BlockShape

    _need_gpu()
    shape = Shape(4, 2, 64, 49, 64, 3, num_layers=2, num_streams=4)
    stats = {}
    worst = run_block_parity(shape, BlockShape(136, 200, weight_std=0.08), 3, stats=stats)
    print("ragged thin block worst |dx|", worst, stats)


@pytest.mark.gpu
@pytest.mark.parametrize("intermediate", [9728, 6144, 4864])
def test_block_wide_tiles_of_the_cooperative_path(intermediate):
    """Two streams of 196 tokens (392 rows: the cooperative GEMM path) and
    hidden 2048.  The gate/up projection (K = 2048) takes one round of tiles
    on a 152-SM GB300 without splitting K, so SiLU(gate) * up is formed in its
    epilogue (each unit holds a block of gate rows and the same up rows): with
    MLP 9728 (N = 19456) 76 x 2 tiles of 256 W rows, with MLP 6144
    (N = 12288) 64 x 2 tiles of 192, with MLP 4864 (N = 9728) 76 x 2 tiles of
    128.  The other projections keep 128-wide tiles and split K."""
    from paper_2605_31598_gb300.inputs import BlockShape

    _need_gpu()
    shape = Shape(16, 2, 128, 196, 256, 3, num_layers=1, num_streams=2)
    stats = {}
    worst = run_block_parity(shape, BlockShape(2048, intermediate), 2, stats=stats)
    print(f"wide-tile block (MLP {intermediate}) worst |dx|", worst, stats)


@pytest.mark.gpu
@pytest.mark.parametrize("streams,tokens", [(1, 196), (2, 16)])
def test_block_multi_layer_call_equals_layer_calls(streams, tokens):
    """One call over every layer (where the thin path computes layer l+1's
    input RMSNorm inside layer l's residual update) gives bit for bit the
    hidden states, states and caches of one call per layer."""
    from paper_2605_31598_gb300.inputs import BlockShape

    _need_gpu()
    shape = Shape(4, 2, 64, tokens, 64, 3, num_layers=3, num_streams=streams)
    block = BlockShape(256, 512, weight_std=0.08)
    bc = statekv_block_config(block.hidden, block.intermediate, block.rms_eps, block.rope_theta,
                              1.0, 0)
    wts = block_weights(shape, block, device="cuda")
    warr = block_weights_array(wts)
    engs = [StateKV(make_config(shape)) for _ in range(2)]
    wss = [torch.empty(e.block_workspace_bytes(bc), dtype=torch.uint8, device="cuda") for e in engs]
    for n in range(1, 4):
        x = block_input(shape, block, n, device="cuda")
        y_all = torch.empty_like(x)
        assert engs[0].block_frame(bc, warr, x, y_all, wss[0]) == 0
        y = x.clone()
        for l in range(shape.num_layers):
            y_next = torch.empty_like(y)
            assert engs[1].block_frame(bc, warr, y, y_next, wss[1], layer_begin=l, layer_count=1) == 0
            y = y_next
        torch.cuda.synchronize()
        assert torch.equal(y_all, y), f"frame {n}"
        for s in range(streams):
            for l in range(shape.num_layers):
                (ka, va, pa, _), (kb, vb, pb, _) = engs[0].state(s, l), engs[1].state(s, l)
                assert torch.equal(pa, pb)
                used = pa >= 0
                assert torch.equal(ka[used], kb[used]) and torch.equal(va[used], vb[used])
                ca, cb = engs[0].cache(s, l), engs[1].cache(s, l)
                assert ca[2].length == cb[2].length == n * tokens
                assert torch.equal(ca[0][:, :n * tokens], cb[0][:, :n * tokens])
                assert torch.equal(ca[1][:, :n * tokens], cb[1][:, :n * tokens])
    assert engs[0].sync() == 0 and engs[1].sync() == 0


@pytest.mark.gpu
def test_block_paired_ctas_ragged_tiles():
    """11 streams of 196 tokens (2156 rows) and widths that leave ragged tiles of
    the CTA-pair GEMM (512 W rows x 160 rows of X): hidden 2112 and 36 heads of 64
    (QKV with bias and down with the residual: 4.1 and 4.5 tiles of W, the last one
    of a single 256-row block), MLP 2112 (8.25 gate/up tiles of 256), 13.5 tiles of
    X (no row of the last tile's second half exists)."""
    from paper_2605_31598_gb300.inputs import BlockShape

    _need_gpu()
    shape = Shape(28, 4, 64, 196, 208, 2, num_layers=1, num_streams=11)
    stats = {}
    worst = run_block_parity(shape, BlockShape(2112, 2112), 2, check_frames=[2], stats=stats)
    print("paired ragged block worst |dx|", worst, stats)


class _GemmPlan(ctypes.Structure):
    """The library's GemmPlan (csrc/statekv_kernels.cuh)."""
    _fields_ = [(n, ctypes.c_int) for n in ("pair_bn", "n_tiles", "m_pairs", "k_steps", "kps",
                                            "splits", "units", "counters")]
    _fields_ += [("partial_bytes", ctypes.c_size_t)]


def _pair_plan(rows, n, k, gate_up=False):
    """(X rows per tile, tiles) of the CTA-pair GEMM for this product; (0, _): not on pairs."""
    plan = statekv.lib()["_ZN7statekv9gemm_planEiiii"]  # statekv::gemm_plan(int, int, int, int)
    plan.restype, plan.argtypes = _GemmPlan, [ctypes.c_int] * 4
    p = plan(rows, n, k, torch.cuda.get_device_properties(0).multi_processor_count)
    per_row = -(-(n // 2) // 256) if gate_up else p.n_tiles
    return p.pair_bn, per_row * (p.units // p.n_tiles)


@pytest.mark.gpu
@pytest.mark.parametrize("streams,tokens,hidden,hq,hkv,d,inter,want", [
    # the narrowest tile; 280 rows
    (2, 140, 2048, 16, 2, 64, 5000, {"gate_up": (96, 60)}),
    # the widest tile, whose ring has three stages, with bias, SiLU and residual
    (11, 205, 3136, 32, 4, 64, 2048,
     {"qkv": (160, 75), "o": (256, 63), "gate_up": (256, 72), "down": (256, 63)}),
    # 76 pairs: a second tile per pair with the residual
    (18, 196, 3136, 32, 4, 64, 2048,
     {"qkv": (256, 70), "o": (192, 133), "gate_up": (192, 152), "down": (192, 133)}),
    # a second tile per pair with bias, on the three-stage ring
    (14, 193, 2048, 32, 8, 128, 2048,
     {"qkv": (256, 132), "o": (160, 68), "gate_up": (160, 136), "down": (160, 68)}),
])
def test_block_on_cta_pairs(streams, tokens, hidden, hq, hkv, d, inter, want):
    """Every tile width of the CTA-pair GEMM not met above, and pairs that take a second
    tile; the plans are those the cases are for (on 152 SMs)."""
    from paper_2605_31598_gb300.inputs import BlockShape

    _need_gpu()
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        rows = streams * tokens
        plans = {"qkv": _pair_plan(rows, (hq + 2 * hkv) * d, hidden), "o": _pair_plan(rows, hidden, hq * d),
                 "gate_up": _pair_plan(rows, 2 * inter, hidden, True), "down": _pair_plan(rows, hidden, inter)}
        assert {k: v for k, v in plans.items() if v[0]} == want
    shape = Shape(hq, hkv, d, tokens, tokens + 12, 2, num_layers=1, num_streams=streams)
    stats = {}
    worst = run_block_parity(shape, BlockShape(hidden, inter), 2, check_frames=[2], stats=stats)
    print(f"pairs {want} worst |dx|", worst, stats)
