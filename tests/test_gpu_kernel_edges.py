"""GPU parity at the sizes where a kernel variant can go wrong: edges of its tiles, remainders, the smallest and largest of its
range.  Every case is compared with the fp64 oracle under the tolerances of util.py."""
import numpy as np
import pytest

from paper_2402_19427_b200 import inputs as synth
from util import assert_close, f64, oracle_prefill, to_dev, to_np

pytestmark = pytest.mark.gpu
GENERIC = 1  # RGLRU_FLAG_FORCE_GENERIC


def forward_and_backward(oracle, B, T, D, H, io, flags, seed, in_place=True):
    """Forward with in-place state and backward through the carried state, both against the oracle."""
    import torch
    from paper_2402_19427_b200 import binding
    inp = synth.make_inputs(B, T, D, H, io=io, seed=seed, with_dy=True, with_state=True, bias_scale=0.2)
    params = binding.Params.from_numpy(inp["params"], io)
    x, h0, cs = to_dev(inp["x"], io), to_dev(inp["h0"]), to_dev(inp["conv_state"], io)
    h, c = (h0.clone(), cs.clone())
    y, _, _ = binding.prefill(x, params, h0=h, conv_state_in=c, h_T=h, conv_state_out=c, flags=flags)
    ws = binding.alloc_workspace(binding.make_shape(B, T, D, H, x.dtype, flags=flags), binding.OP_BACKWARD, x.device)
    ws[256:].fill_(0xFF)   # NaN patterns: nothing may depend on what the workspace held
    g = binding.backward(x, params, to_dev(inp["dy"], io), h0=h0, conv_state_in=cs, flags=flags, state_grads=True, workspace=ws)
    torch.cuda.synchronize()
    assert binding.query_status(ws) == binding.OK
    h064, cs64 = inp["h0"].astype(np.float64), inp["conv_state"].astype(np.float64)
    yr, hr, cr = oracle_prefill(oracle, inp, h0=h064, cs=cs64)
    assert_close("y", to_np(y), yr, io); assert_close("h_T", to_np(h), hr, io)
    assert np.array_equal(to_np(c), cr)
    gr = oracle.backward(inp["x"].astype(np.float64), f64(inp["params"]), H, inp["dy"].astype(np.float64), h0=h064, conv_state_in=cs64, state_grads=True)
    for k in gr:
        # fp32: the 1e-4 bound is absolute for values of order one; gradients that sum over many tokens scale with their size
        scale = max(1.0, float(np.abs(gr[k]).max())) if io == "f32" else 1.0
        assert_close("d" + k, to_np(g[k]), gr[k], io, scale=scale)


@pytest.mark.parametrize("B,T,D,H,io", [
    (2, 321, 1600, 5, "f32"),    # 64-row blocks, six chunks with a one-token tail
    (2, 321, 1610, 5, "f32"),    # the same with a head width that is no multiple of four (322: scalar loads)
    (2, 257, 1610, 5, "bf16"),
    (1, 32, 32, 1, "f32"), (1, 33, 33, 1, "f32"), (3, 65, 132, 2, "f32"),   # 32-row blocks at their edges
    (1, 70, 1024, 1, "f32"),     # the widest head
])
def test_cuda_core_blocks_and_chunk_chain(oracle, B, T, D, H, io):
    forward_and_backward(oracle, B, T, D, H, io, GENERIC, seed=900 + T)


@pytest.mark.parametrize("B,T,Dh,H", [
    (2, 1, 256, 1), (1, 63, 256, 1), (2, 65, 128, 3), (1, 127, 96, 3),   # one chunk, tails, a partial last group of heads
    (1, 1203, 160, 2),    # a long chain of chunks, channels beyond the last 128
    (3, 1030, 64, 5),
])
def test_tensor_core_backward_of_ragged_sequences(oracle, B, T, Dh, H):
    forward_and_backward(oracle, B, T, Dh * H, H, "bf16", 0, seed=700 + T)


@pytest.mark.parametrize("B,T,Dh,H", [
    (2, 77, 352, 2), (3, 1, 288, 1), (1, 64, 320, 3), (1, 200, 1024, 1),   # 3 and 8 channel tiles of a head, the last one part empty
    (1, 515, 544, 1),      # 5 tiles; nine K blocks, the last a half one
    (2, 8300, 288, 1),     # 130 chunks in a chain
])
def test_tensor_core_kernels_of_heads_wider_than_256(oracle, B, T, Dh, H):
    forward_and_backward(oracle, B, T, Dh * H, H, "bf16", 0, seed=300 + T)


def test_wide_heads_with_gate_branch_and_decay_product(oracle):
    import torch
    from paper_2402_19427_b200 import binding
    B, T, D, H = 2, 150, 704, 2
    inp = synth.make_inputs(B, T, D, H, io="bf16", seed=41, with_state=True, with_dy=True)
    params = binding.Params.from_numpy(inp["params"], "bf16")
    ap = torch.empty(B, D, dtype=torch.float32, device="cuda")
    y, hT, _ = binding.prefill(to_dev(inp["x"], "bf16"), params, h0=to_dev(inp["h0"]), gate_branch=to_dev(inp["dy"], "bf16"), a_prod=ap)
    torch.cuda.synchronize()
    branch = inp["dy"].astype(np.float64)
    yr, hr, _, apr = oracle.prefill(inp["x"].astype(np.float64), f64(inp["params"]), H, h0=inp["h0"].astype(np.float64), gate_branch=branch, with_a_prod=True)
    assert_close("y", to_np(y), yr, "bf16"); assert_close("h_T", to_np(hT), hr, "bf16"); assert_close("a_prod", to_np(ap), apr, "bf16")


@pytest.mark.parametrize("B,Dh,H", [(1, 256, 1), (8, 160, 3), (9, 32, 2), (16, 96, 2), (17, 224, 2), (48, 256, 10), (49, 256, 10), (64, 96, 16)])
def test_decode_step_at_the_edges_of_its_two_kernels(oracle, B, Dh, H):
    """Batch tiles of 8 and 16 sequences with remainders, widths that leave a cluster of one to eight blocks, and the batch at
    which the step changes kernels; state in place, biases, several steps."""
    import torch
    from paper_2402_19427_b200 import binding
    T0, steps, D = 2, 3, Dh * H
    inp = synth.make_inputs(B, T0 + steps, D, H, io="bf16", seed=50 + B, bias_scale=0.3)
    params = binding.Params.from_numpy(inp["params"], "bf16")
    x = to_dev(inp["x"], "bf16")
    _, h, cs = binding.prefill(x[:, :T0].contiguous(), params)
    ys = [binding.decode_step(x[:, t].contiguous(), params, h, cs) for t in range(T0, T0 + steps)]
    torch.cuda.synchronize()
    yr, hr, cr = oracle_prefill(oracle, inp)
    assert_close("y", np.stack([to_np(v) for v in ys], 1), yr[:, T0:], "bf16")
    assert_close("h", to_np(h), hr, "bf16")
    assert np.array_equal(to_np(cs), cr)


def test_replayed_graph_of_chained_chunks(oracle):
    """A CUDA graph replays a call with the tags of its capture: records that the first replay left in the workspace must not be
    taken for those of the second, which works on other inputs."""
    import torch
    from paper_2402_19427_b200 import binding
    for io, Dh, flags in (("f32", 64, GENERIC), ("bf16", 288, 0), ("f32", 96, 0), ("f32", 672, 0)):
        B, T, H = 1, 700, 1
        first, second = [synth.make_inputs(B, T, Dh * H, H, io=io, seed=60 + k, with_dy=True) for k in range(2)]
        params = binding.Params.from_numpy(first["params"], io)
        x, dy = to_dev(first["x"], io), to_dev(first["dy"], io)
        shape = binding.make_shape(B, T, Dh * H, H, x.dtype, flags=flags)
        ws, wsb = [binding.alloc_workspace(shape, op, x.device) for op in (binding.OP_PREFILL, binding.OP_BACKWARD)]
        y = torch.empty_like(x)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            binding.prefill(x, params, y=y, workspace=ws, flags=flags)   # first use outside the capture
            binding.backward(x, params, dy, y=y, workspace=wsb, flags=flags)
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                binding.prefill(x, params, y=y, workspace=ws, flags=flags)
                g = binding.backward(x, params, dy, y=y, workspace=wsb, flags=flags)
            graph.replay()
            x.copy_(to_dev(second["x"], io)); dy.copy_(to_dev(second["dy"], io))
            graph.replay()
        torch.cuda.synchronize()
        second["params"] = first["params"]
        yr, _, _ = oracle_prefill(oracle, second)
        gr = oracle.backward(second["x"].astype(np.float64), f64(first["params"]), H, second["dy"].astype(np.float64))
        assert_close("y", to_np(y), yr, io)
        assert_close("dx", to_np(g["x"]), gr["x"], io, scale=max(1.0, float(np.abs(gr["x"]).max())) if io == "f32" else 1.0)


@pytest.mark.parametrize("B,T,Dh,H,merge,keep", [(1, 2000, 256, 1, False, True), (1, 2000, 256, 1, False, False), (1, 700, 96, 2, False, True),
                                                (3, 130, 256, 2, True, True), (1, 1999, 256, 1, True, False), (2, 64, 256, 1, False, True)])
def test_replayed_graph_of_a_time_split_forward(oracle, B, T, Dh, H, merge, keep):
    """The fused prefill with sequences split in time over several CTA pairs: a replay of the captured call must not take the carry
    records that the replay before it left in the workspace for its own.  Every replay works on other inputs."""
    import torch
    from paper_2402_19427_b200 import binding
    D = Dh * H
    rounds = [synth.make_inputs(B, T, D, H, io="bf16", seed=80 + k, with_dy=True, with_state=True) for k in range(4)]
    params = binding.Params.from_numpy(rounds[0]["params"], "bf16")
    x, h0, branch = to_dev(rounds[0]["x"], "bf16"), to_dev(rounds[0]["h0"]), to_dev(rounds[0]["dy"], "bf16") if merge else None
    ws = binding.alloc_workspace(binding.make_shape(B, T, D, H, x.dtype), binding.OP_PREFILL, x.device) if keep else None
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        binding.prefill(x, params, h0=h0, workspace=ws, gate_branch=branch)   # first use outside the capture
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            y, hT, _ = binding.prefill(x, params, h0=h0, workspace=ws, gate_branch=branch)
        for inp in rounds:
            x.copy_(to_dev(inp["x"], "bf16")); h0.copy_(to_dev(inp["h0"]))
            if merge:
                branch.copy_(to_dev(inp["dy"], "bf16"))
            graph.replay()
            stream.synchronize()
            yr, hr, _ = oracle.prefill(inp["x"].astype(np.float64), f64(rounds[0]["params"]), H, h0=inp["h0"].astype(np.float64),
                                       gate_branch=inp["dy"].astype(np.float64) if merge else None)
            assert_close("y", to_np(y), yr, "bf16"); assert_close("h_T", to_np(hT), hr, "bf16")


@pytest.mark.parametrize("change,error", [
    (dict(h0=lambda t: t.double()), ValueError), (dict(x=lambda t: t.transpose(0, 1)), ValueError), (dict(workspace=lambda t: t[:128]), RuntimeError),
    (dict(flags=lambda v: 1 << 40), RuntimeError), (dict(conv_state_in=lambda t: t.cpu()), ValueError)])
def test_calls_the_native_path_does_not_take(change, error):
    """A call with an argument that is wrong raises what the checked path raises, launches nothing, and leaves the next call fine."""
    import torch
    from paper_2402_19427_b200 import binding
    inp = synth.make_inputs(2, 2, 64, 2, io="f32", seed=3, with_state=True)
    params = binding.Params.from_numpy(inp["params"], "f32")
    args = dict(x=to_dev(inp["x"]), h0=to_dev(inp["h0"]), conv_state_in=to_dev(inp["conv_state"]), flags=0,
                workspace=binding.alloc_workspace(binding.make_shape(2, 2, 64, 2, torch.float32), binding.OP_PREFILL, torch.device("cuda", 0)))
    good = binding.prefill(params=params, **args)[0].clone()
    name, make = next(iter(change.items()))
    if name == "flags":   # a flag word wider than 32 bits is truncated as ctypes does, not an error
        assert torch.equal(binding.prefill(params=params, **dict(args, flags=make(0)))[0], good)
        return
    with pytest.raises(error):
        binding.prefill(params=params, **dict(args, **{name: make(args[name])}))
    assert torch.equal(binding.prefill(params=params, **args)[0], good)


def test_a_call_that_fails_in_the_library_is_not_made_twice(oracle, monkeypatch):
    """A batch beyond the launch limits of one of the backward's kernels (more than 65535 sequences) fails after other kernels have been
    launched.  The error is raised by the one call that met it: nothing is launched again, and the next call, which updates state in
    place, neither reports that error nor runs twice."""
    import torch
    from paper_2402_19427_b200 import binding
    B, D = 65536, 32
    inp = synth.make_inputs(1, 1, D, 1, io="bf16", seed=9)
    params = binding.Params.from_numpy(inp["params"], "bf16")
    x = torch.zeros(B, 1, D, dtype=torch.bfloat16, device="cuda")
    ws = binding.alloc_workspace(binding.make_shape(B, 1, D, 1, x.dtype), binding.OP_BACKWARD, x.device)
    step = synth.make_inputs(3, 1, 64, 2, io="f32", seed=10, with_state=True)
    p32 = binding.Params.from_numpy(step["params"], "f32")
    x32, h, cs = to_dev(step["x"][:, 0]), to_dev(step["h0"]), to_dev(step["conv_state"])
    calls = []
    real = binding.load()

    class Counting:
        def __getattr__(self, name):
            if name in ("rglru_backward", "rglru_decode_step"):
                calls.append(name)
            return getattr(real, name)

    monkeypatch.setattr(binding, "load", lambda: Counting())
    with pytest.raises(binding.RglruError) as e:
        binding.backward(x, params, x, workspace=ws)
    assert e.value.code == binding.ERR_CUDA
    y = binding.decode_step(x32, p32, h, cs)
    torch.cuda.synchronize()
    assert calls == []
    yr, hr, cr = oracle_prefill(oracle, step, h0=step["h0"].astype(np.float64), cs=step["conv_state"].astype(np.float64))
    assert_close("y", to_np(y), yr[:, 0], "f32"); assert_close("h", to_np(h), hr, "f32")
    assert np.array_equal(to_np(cs), cr)


def _norm_error(got, ref):
    ref = np.asarray(ref, dtype=np.float64)
    return float(np.linalg.norm(np.asarray(got, dtype=np.float64) - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("B,T,Dh,H", [(2, 203, 96, 3), (1, 130, 256, 1), (1, 64, 288, 2)])
def test_backward_of_ragged_or_wide_layers_is_held_in_fp32(oracle, B, T, Dh, H):
    """bf16 io, fp32 inside: the fp32 gradients are sums of a few hundred to a few ten thousand terms, each rounded a few dozen times at
    2^-24, so their relative 2-norm error stays well below 2^-24 * sqrt(30000) = 1e-5 (measured 1e-6 to 4e-6; 16-bit intermediates
    give 1e-4 to 6e-4)."""
    import torch
    from paper_2402_19427_b200 import binding
    D = Dh * H
    inp = synth.make_inputs(B, T, D, H, io="bf16", seed=70 + T, with_dy=True, with_state=True, bias_scale=0.2)
    params = binding.Params.from_numpy(inp["params"], "bf16")
    x, h0, cs, dy = to_dev(inp["x"], "bf16"), to_dev(inp["h0"]), to_dev(inp["conv_state"], "bf16"), to_dev(inp["dy"], "bf16")
    y, _, _ = binding.prefill(x, params, h0=h0, conv_state_in=cs)
    h064, cs64 = inp["h0"].astype(np.float64), inp["conv_state"].astype(np.float64)
    gr = oracle.backward(inp["x"].astype(np.float64), f64(inp["params"]), H, inp["dy"].astype(np.float64), h0=h064, conv_state_in=cs64, state_grads=True)
    for saved in (None, y):
        g = binding.backward(x, params, dy, h0=h0, conv_state_in=cs, y=saved, state_grads=True)
        torch.cuda.synchronize()
        for k in ("conv_w", "conv_b", "W_a", "b_a", "W_x", "b_x", "lam", "h0"):
            assert _norm_error(to_np(g[k]), gr[k]) < 1e-5, k


@pytest.mark.parametrize("B,T,Dh,H,gain", [(2, 136, 256, 2, 1.0), (1, 2000, 96, 3, 8.0)])
def test_backward_without_the_forward_output_uses_the_forward_kernel(B, T, Dh, H, gain):
    """A forward output that the caller did not keep is the one that the forward would have given him, also where the gate
    pre-activations are large: the gradients are the same bits with it and without it."""
    import torch
    from paper_2402_19427_b200 import binding
    inp = synth.make_inputs(B, T, Dh * H, H, io="bf16", seed=33, with_dy=True, with_state=True, bias_scale=0.2)
    for k in ("W_a", "W_x"):
        inp["params"][k] = inp["params"][k] * gain   # a power of two: still bf16 values
    params = binding.Params.from_numpy(inp["params"], "bf16")
    x, h0, cs, dy = to_dev(inp["x"], "bf16"), to_dev(inp["h0"]), to_dev(inp["conv_state"], "bf16"), to_dev(inp["dy"], "bf16")
    y, _, _ = binding.prefill(x, params, h0=h0, conv_state_in=cs)
    kept = binding.backward(x, params, dy, h0=h0, conv_state_in=cs, y=y, state_grads=True)
    made = binding.backward(x, params, dy, h0=h0, conv_state_in=cs, state_grads=True)
    torch.cuda.synchronize()
    for k in kept:
        assert torch.equal(kept[k], made[k]), k


@pytest.mark.parametrize("B,T,Dh,H,gain", [(2, 203, 352, 2, 1.0), (1, 700, 288, 3, 8.0), (3, 33, 1024, 1, 8.0), (1, 4130, 288, 1, 1.0)])
def test_forward_of_wide_heads_is_held_in_fp32(oracle, B, T, Dh, H, gain):
    """Heads wider than 256, gate pre-activations of order one and of order ten, with channels of long memory: the fp32 outputs are as
    close to the exact ones as fp32 arithmetic comes, 2^-24 * sqrt(30000) = 1e-5 over a thousand steps (measured 1e-6 to 3e-6; 16-bit
    gate products give 1e-4 to 2e-4), and y is the rounded state.  Beyond a thousand steps the rounding of a_t = 0.99999 in the
    channels of long memory adds up like a random walk: the CUDA-core kernel too is 9e-6 off after 9000."""
    import torch
    from paper_2402_19427_b200 import binding
    D = Dh * H
    inp = synth.make_inputs(B, T, D, H, io="bf16", seed=44 + T, with_state=True, bias_scale=0.2)
    p = inp["params"]
    p["W_a"], p["W_x"] = p["W_a"] * gain, p["W_x"] * gain   # a power of two: still bf16 values
    p["lam"][::20] = np.float32(np.log(0.9999 ** 0.125 / (1.0 - 0.9999 ** 0.125)))   # a^c = 0.9999
    params = binding.Params.from_numpy(p, "bf16")
    ap = torch.empty(B, D, dtype=torch.float32, device="cuda")
    y, hT, cso = binding.prefill(to_dev(inp["x"], "bf16"), params, h0=to_dev(inp["h0"]), conv_state_in=to_dev(inp["conv_state"], "bf16"), a_prod=ap)
    torch.cuda.synchronize()
    yr, hr, cr, apr = oracle.prefill(inp["x"].astype(np.float64), f64(p), H, h0=inp["h0"].astype(np.float64), conv_state_in=inp["conv_state"].astype(np.float64), with_a_prod=True)
    assert _norm_error(to_np(hT), hr) < 1e-5 * max(1.0, (T / 1000) ** 0.5)
    assert _norm_error(to_np(y), yr) < 2.0 ** -9   # half a unit in the last of bf16's eight places, at most
    # a product of T factors, each off by up to a few 2^-24: relative to the product itself
    assert np.abs(to_np(ap) - apr).max() <= 4 * T * 2.0 ** -24 * np.abs(apr).max()
    assert np.array_equal(to_np(cso), cr)


def test_wide_heads_do_not_see_one_another(oracle):
    """Block-diagonal gates: a NaN or an infinity in one head's inputs stays in that head, also where a head's width is no multiple of the
    64 channels that the kernels load at once, and in its own sequence."""
    import torch
    from paper_2402_19427_b200 import binding
    B, T, Dh, H = 2, 70, 288, 3
    inp = synth.make_inputs(B, T, Dh * H, H, io="bf16", seed=6)
    params = binding.Params.from_numpy(inp["params"], "bf16")
    x = to_dev(inp["x"], "bf16")
    clean, hc, _ = binding.prefill(x, params)
    bad = x.clone()
    bad[1, 0, Dh] = float("nan"); bad[1, 5, 2 * Dh - 1] = float("inf")   # first and last channel of the middle head, second sequence
    y, hT, _ = binding.prefill(bad, params)
    torch.cuda.synchronize()
    assert torch.isnan(y[1, 0, Dh])
    for h in (0, 2):
        assert torch.equal(y[:, :, h * Dh:(h + 1) * Dh], clean[:, :, h * Dh:(h + 1) * Dh]) and torch.equal(hT[:, h * Dh:(h + 1) * Dh], hc[:, h * Dh:(h + 1) * Dh])
    assert torch.equal(y[0], clean[0]) and torch.equal(hT[0], hc[0])


@pytest.mark.parametrize("B,T,Dh,H", [
    (2, 8, 256, 1), (1, 72, 256, 1), (1, 120, 96, 3),    # one chunk, tails of a chunk, a partial last group of heads
    (1, 1208, 160, 2),                                  # a column shared by many blocks, channels beyond the last 64
    (3, 1032, 64, 5),
])
def test_tensor_core_backward_at_the_edges_of_its_chunks(oracle, B, T, Dh, H):
    """Lengths that are multiples of 8, which the tensor-core backward takes, and of no chunk of 64 tokens."""
    forward_and_backward(oracle, B, T, Dh * H, H, "bf16", 0, seed=720 + T)


def test_replayed_graph_of_the_tensor_core_backward(oracle):
    """Columns shared by several blocks: a replay must not take the records that the replay before it left in the workspace."""
    import torch
    from paper_2402_19427_b200 import binding
    B, T, D, H = 1, 1208, 256, 1
    rounds = [synth.make_inputs(B, T, D, H, io="bf16", seed=90 + k, with_dy=True) for k in range(3)]
    params = binding.Params.from_numpy(rounds[0]["params"], "bf16")
    x, dy = to_dev(rounds[0]["x"], "bf16"), to_dev(rounds[0]["dy"], "bf16")
    ws = binding.alloc_workspace(binding.make_shape(B, T, D, H, x.dtype), binding.OP_BACKWARD, x.device)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        binding.backward(x, params, dy, workspace=ws)   # first use outside the capture
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            g = binding.backward(x, params, dy, workspace=ws)
        for inp in rounds:
            x.copy_(to_dev(inp["x"], "bf16")); dy.copy_(to_dev(inp["dy"], "bf16"))
            graph.replay()
            stream.synchronize()
            gr = oracle.backward(inp["x"].astype(np.float64), f64(rounds[0]["params"]), H, inp["dy"].astype(np.float64))
            for k in ("x", "W_a", "lam"):
                assert_close("d" + k, to_np(g[k]), gr[k], "bf16")


@pytest.mark.parametrize("flags", [0, GENERIC])
def test_many_partial_sums_of_a_wide_layer_are_summed_in_slices(flags):
    """One part for each of 1024 sequences, 5 D = 66560 sums of them.  With zero gate weights and the taps (1, 0, 0, 0) du is dx, so that
    the exact sum is at hand.  All terms are positive: added one after the other they would be off by about 2^-25 sqrt(1024) / 3 = 3.2e-7
    (relative 2-norm), in eight slices by 4e-8."""
    import torch
    from paper_2402_19427_b200 import binding
    B, Dh, H = 1024, 32, 416
    D = Dh * H
    p = synth.make_inputs(1, 1, D, H, io="f32", seed=2)["params"]
    for k in ("W_a", "W_x", "conv_w"):
        p[k][:] = 0.0
    p["conv_w"][0] = 1.0
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    x, dy = torch.randn(B, 1, D, generator=gen, device="cuda"), torch.rand(B, 1, D, generator=gen, device="cuda")
    g = binding.backward(x, binding.Params.from_numpy(p, "f32"), dy, flags=flags)
    assert _norm_error(to_np(g["conv_b"]), g["x"].double().sum((0, 1)).cpu().numpy()) < 2.0 ** -23
