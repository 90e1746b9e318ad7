"""Failure detection on the GPU with a wait that runs out, not a fault.

The watchdog self-test makes the attention kernel's producer wait on a
barrier that nothing completes.  The wait is bounded by the handle's
watchdog: it expires, the kernel records DEVICE_TIMEOUT with the waiting site
in the mapped status word, every warp leaves through its own bounded wait,
and the launch completes.  The handle then reports the error on every call
(sticky), while the CUDA context stays usable for other handles.
"""
import time

import pytest
import torch

from paper_2605_31598_gb300 import StateKV, make_config
from paper_2605_31598_gb300.inputs import WORKLOADS, BlockShape, Shape, batch_qkv, block_weights
from paper_2605_31598_gb300.statekv import SELECTION_LAYER, block_weights_array, statekv_block_config

pytestmark = pytest.mark.gpu

DEVICE_TIMEOUT = 5  # STATEKV_ERR_DEVICE_TIMEOUT


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g

    g.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_expired_wait_is_reported_and_the_context_survives():
    shape = WORKLOADS["toy"]
    eng = StateKV(make_config(shape, watchdog_ms=100))
    t0 = time.monotonic()
    assert eng.watchdog_selftest() == 0
    assert eng.sync() == DEVICE_TIMEOUT
    elapsed = time.monotonic() - t0
    code = eng.device_error()
    assert code & 0xFF == 1, hex(code)  # an attention-kernel wait expired
    assert (code >> 8) & 0xFF == 1, hex(code)  # the self-test's barrier was the first
    assert elapsed < 10.0  # a 100 ms watchdog: the launch ends by itself
    # sticky: the handle refuses further work
    q, k, v = batch_qkv(shape, 1, streams=[0], layers=[0], device="cuda")
    assert eng.prefill_frame(q, k, v, torch.empty_like(q)) == DEVICE_TIMEOUT
    # the context is still usable: a fresh handle runs a frame
    fresh = StateKV(make_config(shape))
    out = torch.full_like(q, float("nan"))
    assert fresh.prefill_frame(q, k, v, out) == 0
    assert fresh.sync() == 0
    assert torch.isfinite(out.float()).all()


@pytest.mark.parametrize("shape,hidden", [
    # one stream: the output projection is the GEMM for few rows
    (Shape(1024, 64, 64, 256, 16384, 3), 128),
    # three streams: it is the one on CTA pairs (51 x 3 tiles of 128 columns fill the SMs)
    (Shape(768, 32, 64, 256, 24320, 3, num_streams=3), 6528),
])
def test_waiting_for_the_previous_kernel_is_not_a_timeout(shape, hidden):
    """The block's output projection is launched programmatically and is in place while
    the selection runs.  Here that takes longer than the watchdog (layer-level scores
    over many heads and a large pool: 1.3 and 1.5 ms against 1 ms, alone), and every kernel
    by itself less than half of it, so a wait may only be timed from the end of the
    selection on.  The results are those of a handle with the default watchdog."""
    block = BlockShape(hidden, 256)
    warr = block_weights_array(weights := block_weights(shape, block, device="cuda"))
    bc = statekv_block_config(block.hidden, block.intermediate, block.rms_eps, block.rope_theta, 1.0, 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(0)
    x = torch.randn((shape.num_streams, shape.tokens_per_frame, hidden), generator=g, device="cuda").bfloat16()
    outs = []
    for ms in (0, 1):
        eng = StateKV(make_config(shape, selection=SELECTION_LAYER, watchdog_ms=ms))
        ws = torch.empty(eng.block_workspace_bytes(bc), dtype=torch.uint8, device="cuda")
        outs.append(torch.full_like(x, float("nan")))
        for _ in range(2):
            assert eng.block_frame(bc, warr, x, outs[-1], ws) == 0
        assert eng.sync() == 0, hex(eng.device_error())
        eng.close()
    assert weights and torch.isfinite(outs[0].float()).all()
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("shape,frames", [
    (Shape(2, 1, 128, 64, 1100, 22), 18),   # one unit of ten key tiles: eight CTAs
    (Shape(6, 3, 64, 37, 1900, 60), 52),    # three units
])
def test_expired_wait_of_a_cluster_is_reported(shape, frames):
    """The self-test on the attention kernel's form for few units over many keys, a
    cluster of CTAs each: every CTA's waits run out, all of them pass the cluster's
    barriers, and the launch ends with the self-test's site."""
    eng = StateKV(make_config(shape, watchdog_ms=100))
    for n in range(1, frames + 1):
        q, k, v = batch_qkv(shape, n, streams=[0], layers=[0], device="cuda")
        assert eng.prefill_frame(q, k, v, torch.empty_like(q)) == 0
    assert eng.sync() == 0
    t0 = time.monotonic()
    assert eng.watchdog_selftest() == 0
    assert eng.sync() == DEVICE_TIMEOUT
    assert time.monotonic() - t0 < 10.0
    code = eng.device_error()
    assert code & 0xFF == 1 and (code >> 8) & 0xFF == 1, hex(code)
    fresh = StateKV(make_config(shape))
    out = torch.full_like(q, float("nan"))
    assert fresh.prefill_frame(q, k, v, out) == 0 and fresh.sync() == 0
    assert torch.isfinite(out.float()).all()
