"""What the parity tests do not show: nothing is written outside the output buffers (guard bytes around every output and
around the workspace), a bounded device-side wait that runs out ends in RGLRU_ERR_TIMEOUT with the context still usable,
and a head shard run on its own reproduces the same channels of the full run bit for bit (Section 4.1: the block-diagonal
gates make heads independent, so tensor-parallel ranks own heads without exchanging anything)."""
import numpy as np
import pytest

from paper_2402_19427_b200 import inputs as synth
from util import Guarded, assert_close, f64, oracle_prefill, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H", [(1, 1, 1), (2, 65, 1), (3, 129, 2), (1, 1000, 1), (8, 320, 3)])
def test_prefill_writes_only_its_outputs(oracle, B, T, H):
    import torch
    from paper_2402_19427_b200 import binding
    D = 256 * H
    inp = synth.make_inputs(B, T, D, H, io="bf16", seed=900 + T, with_state=True)
    params = binding.Params.from_numpy(inp["params"], "bf16")
    x = to_dev(inp["x"], "bf16")
    shape = binding.make_shape(B, T, D, H, torch.bfloat16)
    g = Guarded()
    y = g.empty((B, T, D), torch.bfloat16)
    hT = g.empty((B, D), torch.float32)
    cso = g.empty((B, 3, D), torch.bfloat16)
    ws = g.empty((binding.workspace_bytes(shape, binding.OP_PREFILL),), torch.uint8)
    ws.zero_()
    binding.prefill(x, params, h0=to_dev(inp["h0"]), conv_state_in=to_dev(inp["conv_state"], "bf16"), y=y, h_T=hT,
                    conv_state_out=cso, workspace=ws)
    g.check()
    assert binding.query_status(ws) == binding.OK
    yr, hr, cr = oracle_prefill(oracle, inp, h0=inp["h0"].astype(np.float64), cs=inp["conv_state"].astype(np.float64))
    assert_close("y", to_np(y), yr, "bf16"); assert_close("h_T", to_np(hT), hr, "bf16")
    assert np.array_equal(to_np(cso), cr)


@pytest.mark.parametrize("B,H,flags", [(80, 1, 0), (37, 2, 0), (5, 1, 1)])
def test_decode_step_writes_only_its_outputs(B, H, flags):
    import torch
    from paper_2402_19427_b200 import binding
    D = 256 * H
    inp = synth.make_inputs(B, 4, D, H, io="bf16", seed=77, with_state=True)
    params = binding.Params.from_numpy(inp["params"], "bf16")
    g = Guarded()
    y = g.empty((B, D), torch.bfloat16)
    h = g.empty((B, D), torch.float32); h.copy_(to_dev(inp["h0"]))
    cs = g.empty((B, 3, D), torch.bfloat16); cs.copy_(to_dev(inp["conv_state"], "bf16"))
    shape = binding.make_shape(B, 1, D, H, torch.bfloat16, flags=flags)
    ws = g.empty((binding.workspace_bytes(shape, binding.OP_DECODE),), torch.uint8); ws.zero_()
    for t in range(3):
        binding.decode_step(to_dev(inp["x"][:, t], "bf16"), params, h, cs, y=y, workspace=ws, flags=flags)
    g.check()
    assert torch.isfinite(y.float()).all() and torch.isfinite(h).all()


@pytest.mark.parametrize("B,T,H,io,flags", [(2, 64, 1, "bf16", 0), (1, 200, 2, "bf16", 0), (2, 70, 2, "f32", 1)])
def test_backward_writes_only_its_outputs(B, T, H, io, flags):
    import torch
    from paper_2402_19427_b200 import binding
    D = (256 if io == "bf16" else 32) * H
    dt = torch.bfloat16 if io == "bf16" else torch.float32
    inp = synth.make_inputs(B, T, D, H, io=io, seed=55, with_dy=True)
    params = binding.Params.from_numpy(inp["params"], io)
    x = to_dev(inp["x"], io); dy = to_dev(inp["dy"], io)
    Dh = D // H
    g = Guarded()
    f32 = torch.float32
    out = dict(x=g.empty((B, T, D), dt), conv_w=g.empty((4, D), f32), conv_b=g.empty((D,), f32), W_a=g.empty((H, Dh, Dh), f32),
               b_a=g.empty((D,), f32), W_x=g.empty((H, Dh, Dh), f32), b_x=g.empty((D,), f32), lam=g.empty((D,), f32))
    shape = binding.make_shape(B, T, D, H, dt, flags=flags)
    ws = g.empty((binding.workspace_bytes(shape, binding.OP_BACKWARD),), torch.uint8); ws.zero_()
    binding.backward(x, params, dy, flags=flags, workspace=ws, out=out)
    g.check()
    for k, v in out.items():
        assert torch.isfinite(v.float()).all(), k


def test_a_wait_that_runs_out_is_reported_and_the_next_call_is_clean(oracle):
    """One sequence split in time over several CTA pairs: every tile after the first waits for carry records.  Under the
    test flag the records it looks for never appear, the wait limit is one millisecond, so the kernel gives up, drains and
    returns; the status word says so, and the same workspace then serves an ordinary call that matches the oracle."""
    import torch
    from paper_2402_19427_b200 import binding
    B, T, H = 1, 1024, 1
    inp = synth.make_inputs(B, T, 256 * H, H, io="bf16", seed=13)
    params = binding.Params.from_numpy(inp["params"], "bf16")
    x = to_dev(inp["x"], "bf16")
    shape = binding.make_shape(B, T, 256 * H, H, torch.bfloat16)
    ws = binding.alloc_workspace(shape, binding.OP_PREFILL, x.device)
    prev = binding.set_wait_limit_ns(1_000_000)
    try:
        binding.prefill(x, params, workspace=ws, flags=binding.FLAG_TEST_CARRY_NEVER_ARRIVES)
        torch.cuda.synchronize()
        assert binding.query_status(ws) == binding.ERR_TIMEOUT
        assert binding.query_status(ws) == binding.OK          # reported once
    finally:
        binding.set_wait_limit_ns(prev)
    y, hT, cso = binding.prefill(x, params, workspace=ws)
    torch.cuda.synchronize()
    assert binding.query_status(ws) == binding.OK
    yr, hr, cr = oracle_prefill(oracle, inp)
    assert_close("y", to_np(y), yr, "bf16"); assert_close("h_T", to_np(hT), hr, "bf16")
    assert np.array_equal(to_np(cso), cr)


def test_head_shard_reproduces_the_full_run_bit_for_bit():
    """Heads [1, 3) of a four-head layer run as their own two-head problem on the sliced tensors (what a tensor-parallel
    rank owning those heads would do).  Sequences are dealt whole to the CTA pairs in both runs, so the arithmetic per
    channel is the same and the results must be identical bits."""
    import torch
    from paper_2402_19427_b200 import binding
    B, T, H = 16, 200, 4
    inp = synth.make_inputs(B, T, 256 * H, H, io="bf16", seed=21, with_state=True, bias_scale=0.3)
    params = binding.Params.from_numpy(inp["params"], "bf16")
    y, hT, cso = binding.prefill(to_dev(inp["x"], "bf16"), params, h0=to_dev(inp["h0"]),
                                 conv_state_in=to_dev(inp["conv_state"], "bf16"))
    heads = [1, 2]
    sl = synth.head_slice(inp, heads)
    ch = np.arange(256 * heads[0], 256 * (heads[-1] + 1))
    ps = binding.Params.from_numpy(sl["params"], "bf16")
    ys, hs, cs = binding.prefill(to_dev(sl["x"], "bf16"), ps, h0=to_dev(inp["h0"][:, ch]),
                                 conv_state_in=to_dev(inp["conv_state"][:, :, ch], "bf16"))
    torch.cuda.synchronize()
    chd = torch.from_numpy(ch).to(y.device)
    assert torch.equal(ys, y[:, :, chd]) and torch.equal(hs, hT[:, chd]) and torch.equal(cs, cso[:, :, chd])


def _long_decode(binding, torch, blocks):
    """A CUDA-core decode step of `blocks` blocks of 102 KB of shared memory that each hold an SM for some hundred microseconds."""
    D = 1024
    inp = synth.make_inputs(1, 1, D, 1, io="f32", seed=3)
    params = binding.Params.from_numpy(inp["params"], "f32")
    B = 16 * blocks
    x, h, cs, y = torch.zeros(B, D, device="cuda"), torch.zeros(B, D, device="cuda"), torch.zeros(B, 3, D, device="cuda"), torch.empty(B, D, device="cuda")
    ws = binding.alloc_workspace(binding.make_shape(B, 1, D, 1, torch.float32), binding.OP_DECODE, x.device)
    return lambda: binding.decode_step(x, params, h, cs, y=y, workspace=ws)


@pytest.mark.parametrize("merge", [False, True])
def test_a_time_split_forward_waits_for_sms_that_other_work_holds(oracle, merge):
    """Sequences split in time over CTA pairs that need 128 SMs, while a kernel on another stream keeps most of the 148 for several times the
    wait limit: the pairs that run wait for those that cannot start yet, and the call ends as it would have done alone."""
    import torch
    from paper_2402_19427_b200 import binding
    B, T, H = 1, 2048, 4
    inp = synth.make_inputs(B, T, 256 * H, H, io="bf16", seed=29, with_dy=True)
    params = binding.Params.from_numpy(inp["params"], "bf16")
    x, branch = to_dev(inp["x"], "bf16"), to_dev(inp["dy"], "bf16") if merge else None
    ws = binding.alloc_workspace(binding.make_shape(B, T, 256 * H, H, torch.bfloat16), binding.OP_PREFILL, x.device)
    hold = _long_decode(binding, torch, 140)
    call = lambda: binding.prefill(x, params, workspace=ws, gate_branch=branch)
    s0, s1 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s0):
        hold()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(); hold(); e1.record()
    torch.cuda.synchronize()
    held_ns = int(e0.elapsed_time(e1) * 1e6)
    with torch.cuda.stream(s1):
        call()
    torch.cuda.synchronize()
    prev = binding.set_wait_limit_ns(held_ns // 5)
    try:
        with torch.cuda.stream(s0):
            hold()
        with torch.cuda.stream(s1):
            y, hT, _ = call()
        torch.cuda.synchronize()
        assert binding.query_status(ws) == binding.OK
    finally:
        binding.set_wait_limit_ns(prev)
    yr, hr, _, _ = oracle.prefill(inp["x"].astype(np.float64), f64(inp["params"]), H, gate_branch=inp["dy"].astype(np.float64) if merge else None, with_a_prod=True)
    assert_close("y", to_np(y), yr, "bf16"); assert_close("h_T", to_np(hT), hr, "bf16")


def test_time_split_forwards_on_two_streams(oracle):
    """Two time-split prefills in flight at once, each wanting most of the GPU, round after round: both finish and match the oracle."""
    import torch
    from paper_2402_19427_b200 import binding
    runs = []
    for k, (T, H) in enumerate(((2048, 4), (1500, 5))):
        inp = synth.make_inputs(1, T, 256 * H, H, io="bf16", seed=31 + k)
        x = to_dev(inp["x"], "bf16")
        ws = binding.alloc_workspace(binding.make_shape(1, T, 256 * H, H, torch.bfloat16), binding.OP_PREFILL, x.device)
        runs.append((inp, binding.Params.from_numpy(inp["params"], "bf16"), x, ws, torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _ in range(20):
        out = []
        for _, params, x, ws, st in runs:
            with torch.cuda.stream(st):
                out.append(binding.prefill(x, params, workspace=ws))
    torch.cuda.synchronize()
    for (inp, _, _, ws, _), (y, hT, _) in zip(runs, out):
        assert binding.query_status(ws) == binding.OK
        yr, hr, _ = oracle_prefill(oracle, inp)
        assert_close("y", to_np(y), yr, "bf16"); assert_close("h_T", to_np(hT), hr, "bf16")


def test_other_python_threads_run_while_a_launch_blocks():
    """A launch into a full queue blocks until the GPU has taken some of it.  The call has given up the interpreter lock by then, so a
    second Python thread goes on at its own pace."""
    import threading
    import time
    import torch
    from paper_2402_19427_b200 import binding
    inp = synth.make_inputs(2, 1, 64, 2, io="f32", seed=4, with_state=True)
    params = binding.Params.from_numpy(inp["params"], "f32")
    x, h, cs = to_dev(inp["x"][:, 0]), to_dev(inp["h0"]), to_dev(inp["conv_state"])
    y = torch.empty_like(x)
    ws = binding.alloc_workspace(binding.make_shape(2, 1, 64, 2, torch.float32), binding.OP_DECODE, x.device)
    step = lambda: binding.decode_step(x, params, h, cs, y=y, workspace=ws)
    step()
    torch.cuda.synchronize()
    gaps, stop = [], threading.Event()

    def tick():
        last = time.perf_counter()
        while not stop.is_set():
            time.sleep(0.002)
            now = time.perf_counter()
            gaps.append(now - last)
            last = now

    worker = threading.Thread(target=tick)
    worker.start()
    torch.cuda._sleep(1_000_000_000)   # about half a second of GPU time in front of the queue
    longest = 0.0
    for _ in range(4000):
        t = time.perf_counter()
        step()
        longest = max(longest, time.perf_counter() - t)
    stop.set()
    worker.join()
    torch.cuda.synchronize()
    assert longest > 0.1, "no launch blocked: the queue took all of them"
    assert max(gaps) < 0.5 * longest, (max(gaps), longest)


@pytest.mark.parametrize("B,T,Dh,H,io,flags,backward", [
    (1, 700, 64, 2, "f32", 1, False), (1, 700, 64, 2, "f32", 1, True),          # chunk chains of the CUDA-core kernels
    (1, 2000, 288, 1, "bf16", 0, False), (1, 700, 64, 2, "f32", 0, False), (4, 1300, 64, 4, "f32", 0, False), (1, 200, 1024, 1, "f32", 0, False),   # split forwards
    (1, 700, 64, 2, "f32", 0, True), (4, 1300, 64, 4, "f32", 0, True), (1, 701, 96, 2, "bf16", 0, True), (1, 300, 288, 2, "bf16", 0, "saved"),     # and backwards
    (1, 2000, 256, 1, "bf16", 0, True), (1, 2000, 256, 1, "bf16", 0, "saved"),  # blocks that share a column of the 16-bit reverse scan; the forward in front of it
])
def test_every_wait_for_a_carry_is_bounded(oracle, B, T, Dh, H, io, flags, backward):
    """As above for the other kernels that hand carries from block to block: the wait runs out, the status says so, once, and the next
    call on the same workspace is right."""
    import torch
    from paper_2402_19427_b200 import binding
    D = Dh * H
    inp = synth.make_inputs(B, T, D, H, io=io, seed=14, with_dy=True)
    params = binding.Params.from_numpy(inp["params"], io)
    x, dy = to_dev(inp["x"], io), to_dev(inp["dy"], io)
    ws = binding.alloc_workspace(binding.make_shape(B, T, D, H, x.dtype, flags=flags), binding.OP_BACKWARD if backward else binding.OP_PREFILL, x.device)
    y = binding.prefill(x, params, flags=flags)[0] if backward == "saved" else None

    def call(f):
        return binding.backward(x, params, dy, y=y, flags=f, workspace=ws)["x"] if backward else binding.prefill(x, params, flags=f, workspace=ws)[0]

    call(flags)
    prev = binding.set_wait_limit_ns(1_000_000)
    try:
        call(flags | binding.FLAG_TEST_CARRY_NEVER_ARRIVES)
        torch.cuda.synchronize()
        assert binding.query_status(ws) == binding.ERR_TIMEOUT
        assert binding.query_status(ws) == binding.OK
    finally:
        binding.set_wait_limit_ns(prev)
    out = call(flags)
    torch.cuda.synchronize()
    assert binding.query_status(ws) == binding.OK
    ref = oracle.backward(inp["x"].astype(np.float64), f64(inp["params"]), H, inp["dy"].astype(np.float64))["x"] if backward else oracle_prefill(oracle, inp)[0]
    assert_close("out", to_np(out), ref, io, scale=max(1.0, float(np.abs(ref).max())) if io == "f32" else 1.0)


@pytest.mark.parametrize("flags", [0, 1])   # split products, CUDA cores
def test_a_failed_link_ends_the_chain_at_once(flags):
    """2000 chunks in a chain, of which the GPU holds less than a quarter at a time: a link that gives up tells the next, so the call ends
    after one wait limit and not after one per wave of blocks."""
    import time
    import torch
    from paper_2402_19427_b200 import binding
    T, D = 128000, 64
    inp = synth.make_inputs(1, 1, D, 1, io="f32", seed=15)
    params = binding.Params.from_numpy(inp["params"], "f32")
    x = torch.zeros(1, T, D, device="cuda")
    ws = binding.alloc_workspace(binding.make_shape(1, T, D, 1, torch.float32, flags=flags), binding.OP_PREFILL, x.device)
    y = torch.empty_like(x)
    binding.prefill(x, params, y=y, workspace=ws, flags=flags)
    torch.cuda.synchronize()
    limit = 0.1
    prev = binding.set_wait_limit_ns(int(limit * 1e9))
    try:
        t = time.perf_counter()
        binding.prefill(x, params, y=y, workspace=ws, flags=flags | binding.FLAG_TEST_CARRY_NEVER_ARRIVES)
        torch.cuda.synchronize()
        t = time.perf_counter() - t
        assert binding.query_status(ws) == binding.ERR_TIMEOUT
    finally:
        binding.set_wait_limit_ns(prev)
    assert limit < t < 2 * limit, t


@pytest.mark.parametrize("B,T,Dh,H,io,merge", [
    (2, 70, 96, 3, "bf16", False), (1, 130, 160, 3, "bf16", True), (3, 33, 32, 9, "bf16", False),   # partial last groups, unused channel slots
    (2, 71, 288, 2, "bf16", True), (1, 4100, 288, 1, "bf16", False),                                # split products: heads wider than 256,
    (2, 150, 96, 3, "f32", True), (3, 705, 64, 7, "f32", False), (1, 131, 672, 1, "f32", True),     # fp32, blocks of 32 and 64 tokens, three sets of accumulators
    (2, 67, 34, 3, "bf16", False), (1, 97, 66, 2, "f32", True),                                     # CUDA-core kernels, odd widths
])
def test_prefill_of_other_widths_writes_only_its_outputs(oracle, B, T, Dh, H, io, merge):
    import torch
    from paper_2402_19427_b200 import binding
    D, dt = Dh * H, torch.bfloat16 if io == "bf16" else torch.float32
    inp = synth.make_inputs(B, T, D, H, io=io, seed=910 + T, with_state=True, with_dy=True)
    params = binding.Params.from_numpy(inp["params"], io)
    g = Guarded()
    y, hT, cso, ap = g.empty((B, T, D), dt), g.empty((B, D), torch.float32), g.empty((B, 3, D), dt), g.empty((B, D), torch.float32)
    ws = g.empty((binding.workspace_bytes(binding.make_shape(B, T, D, H, dt), binding.OP_PREFILL),), torch.uint8)
    ws[:256].zero_()
    binding.prefill(to_dev(inp["x"], io), params, h0=to_dev(inp["h0"]), conv_state_in=to_dev(inp["conv_state"], io), y=y, h_T=hT, conv_state_out=cso,
                    workspace=ws, a_prod=ap, gate_branch=to_dev(inp["dy"], io) if merge else None)
    g.check()
    assert binding.query_status(ws) == binding.OK
    yr, hr, cr, apr = oracle.prefill(inp["x"].astype(np.float64), f64(inp["params"]), H, h0=inp["h0"].astype(np.float64),
                                     conv_state_in=inp["conv_state"].astype(np.float64), gate_branch=inp["dy"].astype(np.float64) if merge else None, with_a_prod=True)
    assert_close("y", to_np(y), yr, io); assert_close("h_T", to_np(hT), hr, io); assert_close("a_prod", to_np(ap), apr, io)
    assert np.array_equal(to_np(cso), cr)


@pytest.mark.parametrize("B,T,Dh,H,io,saved", [
    (2, 72, 96, 3, "bf16", True), (1, 136, 160, 3, "bf16", False), (3, 40, 32, 9, "bf16", True),   # tensor cores: partial groups, tails of a chunk
    (2, 71, 96, 3, "bf16", True), (1, 64, 288, 2, "bf16", False), (2, 67, 34, 3, "f32", False),    # ragged, wide, odd widths
    (2, 67, 96, 3, "f32", True), (3, 705, 64, 7, "f32", False), (1, 131, 672, 1, "f32", False),    # fp32
])
def test_backward_of_other_shapes_writes_only_its_outputs(B, T, Dh, H, io, saved):
    import torch
    from paper_2402_19427_b200 import binding
    D, dt, f32 = Dh * H, torch.bfloat16 if io == "bf16" else torch.float32, torch.float32
    inp = synth.make_inputs(B, T, D, H, io=io, seed=56, with_dy=True, with_state=True)
    params = binding.Params.from_numpy(inp["params"], io)
    x, dy, h0, cs = to_dev(inp["x"], io), to_dev(inp["dy"], io), to_dev(inp["h0"]), to_dev(inp["conv_state"], io)
    y = binding.prefill(x, params, h0=h0, conv_state_in=cs)[0] if saved else None
    g = Guarded()
    out = dict(x=g.empty((B, T, D), dt), conv_w=g.empty((4, D), f32), conv_b=g.empty((D,), f32), W_a=g.empty((H, Dh, Dh), f32), b_a=g.empty((D,), f32),
               W_x=g.empty((H, Dh, Dh), f32), b_x=g.empty((D,), f32), lam=g.empty((D,), f32), h0=g.empty((B, D), f32), conv_state=g.empty((B, 3, D), dt))
    ws = g.empty((binding.workspace_bytes(binding.make_shape(B, T, D, H, dt), binding.OP_BACKWARD),), torch.uint8)
    ws[:256].zero_()
    binding.backward(x, params, dy, h0=h0, conv_state_in=cs, y=y, workspace=ws, out=out, state_grads=True, dh_T=h0, dconv_state_out=cs)
    g.check()
    ref = binding.backward(x, params, dy, h0=h0, conv_state_in=cs, y=y, state_grads=True, dh_T=h0, dconv_state_out=cs)
    torch.cuda.synchronize()
    for k, v in out.items():
        assert torch.equal(v, ref[k]), k   # and every element of them is written: the guarded buffers started as 0xA5
