"""The work that a user of this package has it do, as cases that can be timed.

A case is one call (or one forward with its backward) through ``paper_2402_19427_b200.binding``:

* ``prefill``  -- the forward over whole sequences: prompts, training batches, long documents, segments that continue a
  carried state, and the forward merged with the GeLU branch of the recurrent block;
* ``decode``   -- one token for each of B sequences, state updated in place;
* ``backward`` -- the gradients of the forward, for whole training sequences and for segments of truncated back-propagation;
* ``step``     -- forward and backward in fp32, what the small exact runs (gradient checks, reference runs) do.

Widths and head counts are those of ``inputs.CONFIGS``, ``bench.py`` and the tests: D_RNN 2560 as 10 heads of 256 or 16 blocks
of 160, 4096 as 16 heads of 256, 1536 / 2048 as 16 blocks of 96 / 128, 1024 as 4 heads of 256, and 16 blocks of 352 as a
layer whose heads are wider than 256.
"""
from __future__ import annotations

import torch

from paper_2402_19427_b200 import binding

# (D_RNN, heads) of the layers a bf16 case may have, and of the small fp32 ones
LAYERS = [(1024, 4), (1536, 16), (2048, 16), (2560, 10), (2560, 16), (4096, 16)]
WIDE_LAYERS = [(5632, 16)]
F32_LAYERS = [(256, 2), (512, 4), (1024, 4), (1024, 8)]


def _case(op, B, T, D, H, io="bf16", state=False, bias=False, merge=False, keep_y=True, keep_workspace=True, long_memory=False):
    return dict(op=op, B=B, T=T, D=D, H=H, io=io, state=state, bias=bias, merge=merge, keep_y=keep_y,
                keep_workspace=keep_workspace, long_memory=long_memory)


def listed():
    def named(name, *args, **kw):
        return dict(_case(*args, **kw), name=name)

    return [
        # one user's next token: the smallest call there is, latency and host path
        named("decode_one", "decode", 1, 1, 2560, 10),
        # a full serving batch, the batched-decode workload
        named("decode_batch", "decode", 512, 1, 2560, 10),
        # a short prompt of odd length, called the plain way (the call makes its own workspace)
        named("prefill_prompt", "prefill", 1, 197, 2560, 10, keep_workspace=False),
        # the training-shape forward, bench.py's headline workload
        named("prefill_train", "prefill", 8, 2048, 2560, 10),
        # one long document with a share of long-memory channels
        named("prefill_long", "prefill", 1, 65536, 4096, 16, long_memory=True),
        # a ragged segment that continues carried state, 16 blocks of width 160, biases that a trained layer has
        named("prefill_segment", "prefill", 3, 1213, 2560, 16, state=True, bias=True),
        # the forward with the second branch of the block merged in, and the decay product
        named("prefill_merge", "prefill", 8, 2048, 2560, 10, merge=True),
        # heads wider than 256
        named("prefill_wide", "prefill", 2, 777, 5632, 16),
        # the training backward with the forward output saved
        named("backward_train", "backward", 4, 4096, 4096, 16),
        # a ragged segment of truncated back-propagation through time: state gradients, forward output not kept
        named("backward_segment", "backward", 5, 1021, 1536, 16, state=True, bias=True, keep_y=False),
        # the tiny fp32 workload of the parity checks, forward and backward
        named("f32_tiny_step", "step", 1, 256, 256, 2, io="f32"),
        # the largest fp32 run in use
        named("f32_step", "step", 4, 1024, 1024, 4, io="f32", bias=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    op = rng.choices(["decode", "prefill", "backward", "step"], [3, 5, 3, 1])[0]
    if op == "step":
        D, H = rng.choice(F32_LAYERS)
        return _case("step", rng.randint(1, 4), _log_int(rng, 16, 1024), D, H, io="f32", state=rng.random() < 0.3, bias=rng.random() < 0.5)
    wide = rng.random() < 0.1
    D, H = rng.choice(WIDE_LAYERS if wide else LAYERS)
    bias, state, keep_workspace = rng.random() < 0.5, rng.random() < 0.4, rng.random() < 0.8
    if op == "decode":
        return _case("decode", _log_int(rng, 1, 512), 1, D, H, bias=bias, keep_workspace=keep_workspace)
    most_tokens = 2 * 777 if wide else (65536 * 4096 if op == "prefill" else 4 * 4096 * 4096) // D
    B = rng.randint(1, 2 if wide else 8)
    T = _log_int(rng, 32, min(most_tokens // B, 65536 if op == "prefill" else 4096))
    if rng.random() < 0.5 and T >= 128:
        T = T // 128 * 128   # training lengths are round; prompts and segments are not
    if op == "prefill":
        return _case("prefill", B, T, D, H, state=state, bias=bias, merge=rng.random() < 0.2, keep_workspace=keep_workspace, long_memory=rng.random() < 0.3)
    return _case("backward", B, T, D, H, state=state, bias=bias, keep_y=rng.random() < 0.7, keep_workspace=keep_workspace)


class _State:
    """What a program holds before the call: the layer's parameters, this call's tensors and the workspaces it keeps."""


def _dtype(case):
    return torch.bfloat16 if case["io"] == "bf16" else torch.float32


def prepare(case, seed):
    B, T, D, H = case["B"], case["T"], case["D"], case["H"]
    dh, io, dev = D // H, _dtype(case), torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)

    def normal(*shape, scale=1.0, dtype=torch.float32):
        return (torch.randn(*shape, generator=gen, device=dev) * scale).to(dtype)

    s = _State()
    s.case = dict(case)
    # Section 2.4: LeCun-normal gate weights, a^c uniform in [0.9, 0.999]
    conv_w = normal(4, D, scale=0.5, dtype=io)
    W_a, W_x = normal(H, dh, dh, scale=dh ** -0.5, dtype=io), normal(H, dh, dh, scale=dh ** -0.5, dtype=io)
    a_pow_c = 0.9 + 0.099 * torch.rand(D, generator=gen, device=dev, dtype=torch.float64)
    if case["long_memory"]:
        a_pow_c[torch.rand(D, generator=gen, device=dev) < 0.05] = 0.9999
    lam = torch.logit(a_pow_c ** 0.125).float()
    scale = 0.2 if case["bias"] else 0.0
    s.params = binding.Params(conv_w, normal(D, scale=scale), W_a, normal(D, scale=scale), W_x, normal(D, scale=scale), lam)
    if case["op"] == "decode":
        s.x = normal(B, D, dtype=io)
        s.h, s.conv_state = normal(B, D), normal(B, 3, D, dtype=io)
        s.y = torch.empty_like(s.x)
        s.ws = _workspace(case, binding.OP_DECODE, dev)
        return s
    s.x = normal(B, T, D, dtype=io)
    s.h0 = normal(B, D) if case["state"] else None
    s.cs = normal(B, 3, D, dtype=io) if case["state"] else None
    s.ws = _workspace(case, binding.OP_PREFILL, dev)
    if case["op"] == "prefill":
        s.branch = normal(B, T, D, dtype=io) if case["merge"] else None
        s.a_prod = torch.empty(B, D, dtype=torch.float32, device=dev) if case["merge"] else None
        return s
    s.dy = normal(B, T, D, dtype=io)
    s.dh_T = normal(B, D) if case["state"] else None
    s.dcs = normal(B, 3, D, dtype=io) if case["state"] else None
    s.ws_back = _workspace(case, binding.OP_BACKWARD, dev)
    s.y = None
    if case["op"] == "backward":
        if case["keep_y"]:
            s.y = binding.prefill(s.x, s.params, h0=s.h0, conv_state_in=s.cs, workspace=s.ws)[0]
        s.ws = None
    return s


def _workspace(case, op, dev):
    if not case["keep_workspace"]:
        return None
    return binding.alloc_workspace(binding.make_shape(case["B"], case["T"], case["D"], case["H"], _dtype(case)), op, dev)


def run(s):
    c = s.case
    if c["op"] == "decode":
        binding.decode_step(s.x, s.params, s.h, s.conv_state, y=s.y, workspace=s.ws)
        return s.y, s.h, s.conv_state
    if c["op"] == "prefill":
        y, h_T, cs = binding.prefill(s.x, s.params, h0=s.h0, conv_state_in=s.cs, workspace=s.ws, gate_branch=s.branch, a_prod=s.a_prod)
        return (y, h_T, cs) if s.a_prod is None else (y, h_T, cs, s.a_prod)
    out = []
    y = s.y
    if c["op"] == "step":
        out = list(binding.prefill(s.x, s.params, h0=s.h0, conv_state_in=s.cs, workspace=s.ws))
        y = out[0]
    grads = binding.backward(s.x, s.params, s.dy, h0=s.h0, conv_state_in=s.cs, y=y, workspace=s.ws_back, dh_T=s.dh_T,
                             dconv_state_out=s.dcs, state_grads=c["state"])
    return out, grads


def work(case):
    """Bytes: every input and output once, the parameters and their gradients once.  Operations: the gate products (4 D_h per
    element forward, 12 backward: z again, du, dW), the Conv1D and the element-wise part."""
    B, T, D, H = case["B"], case["T"], case["D"], case["H"]
    dh, io = D // H, 2 if case["io"] == "bf16" else 4
    elements = B * T * D
    params = (4 * D + 2 * D * dh) * io + 4 * D * 4
    state = B * D * (4 + 3 * io)
    forward = {"bytes": elements * io * (3 if case["merge"] else 2) + params + state * (2 if case["state"] or case["op"] == "decode" else 1),
               "flops": elements * (4 * dh + 30)}
    if case["merge"]:
        forward["bytes"] += B * D * 4
    if case["op"] in ("prefill", "decode"):
        return forward
    reads_y = case["op"] == "step" or case["keep_y"]
    backward = {"bytes": elements * io * (4 if reads_y else 3) + params + (5 * D + 2 * D * dh + 3 * D) * 4 + (3 * state if case["state"] else 0),
                "flops": elements * (12 * dh + 90)}
    if case["op"] == "backward":
        return backward
    return {k: forward[k] + backward[k] for k in forward}


def tolerance(case):
    # bf16 io keeps 8 significant bits (2^-9 relative per rounding, more where the terms of a sum cancel); fp32 sums of up to a
    # few thousand terms in another order
    if case["io"] == "bf16":
        return {"rel": 1e-2, "max": 5e-2}
    return {"rel": 1e-5, "max": 4e-4}
