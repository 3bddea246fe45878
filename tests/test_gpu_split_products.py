"""GPU parity of the kernels that keep fp32 accuracy on the tensor cores (operands as sums of bf16 values), at the edges of their tiles:
blocks of 32 or 64 tokens and 128 channels, K blocks of 64 (32 in a last half one), segments of eight tokens, splits of dW."""
import numpy as np
import pytest

from paper_2402_19427_b200 import inputs as synth
from test_gpu_kernel_edges import _norm_error, forward_and_backward
from util import assert_close, f64, oracle_prefill, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,Dh,H,io", [
    (1, 1, 32, 1, "f32"), (2, 8, 64, 1, "f32"), (1, 31, 96, 2, "f32"), (3, 33, 128, 2, "f32"), (1, 65, 160, 3, "f32"),   # 32-token blocks
    (4, 640, 256, 4, "f32"), (3, 641, 128, 8, "f32"), (16, 63, 96, 12, "f32"),                                           # 64-token blocks
    (1, 70, 1024, 1, "f32"), (1, 40, 544, 2, "f32"),                                                                     # many channel and K blocks
    (1, 3, 32, 3, "bf16"), (2, 129, 224, 2, "bf16"), (7, 321, 96, 16, "bf16"), (1, 90, 384, 2, "bf16"), (5, 64, 288, 16, "bf16"),
])
def test_split_products_at_the_edges_of_their_tiles(oracle, B, T, Dh, H, io):
    forward_and_backward(oracle, B, T, Dh * H, H, io, 0, seed=300 + T)


@pytest.mark.parametrize("io,B,T,Dh,H", [
    ("f32", 2, 515, 256, 2), ("f32", 1, 1024, 96, 3), ("bf16", 2, 1021, 96, 4), ("bf16", 1, 300, 352, 2),
    ("f32", 2, 300, 160, 2), ("f32", 2, 300, 352, 2), ("f32", 1, 400, 544, 1), ("f32", 1, 400, 1024, 1), ("f32", 40, 64, 512, 2),
    ("f32", 40, 64, 1024, 1), ("bf16", 1, 301, 512, 1), ("bf16", 1, 300, 1024, 1)])
def test_split_products_are_as_exact_as_the_cuda_cores(oracle, io, B, T, Dh, H):
    """No fp32 output is further from the exact one (relative 2-norm) than the CUDA-core kernels' own; the bf16 ones are roundings of such
    values, of which a few fall to the other neighbour."""
    import torch
    from paper_2402_19427_b200 import binding
    inp = synth.make_inputs(B, T, Dh * H, H, io=io, seed=81, with_dy=True, with_state=True, bias_scale=0.2)
    params = binding.Params.from_numpy(inp["params"], io)
    x, h0, cs, dy = to_dev(inp["x"], io), to_dev(inp["h0"]), to_dev(inp["conv_state"], io), to_dev(inp["dy"], io)
    h064, cs64 = inp["h0"].astype(np.float64), inp["conv_state"].astype(np.float64)
    ref = oracle.backward(inp["x"].astype(np.float64), f64(inp["params"]), H, inp["dy"].astype(np.float64), h0=h064, conv_state_in=cs64, state_grads=True)
    if io == "f32" or Dh > 256:   # narrower bf16 heads have another forward
        ref["y"], ref["h_T"], _ = oracle_prefill(oracle, inp, h0=h064, cs=cs64)
    err = []
    for flags in (0, 1):   # 1: RGLRU_FLAG_FORCE_GENERIC
        g = binding.backward(x, params, dy, h0=h0, conv_state_in=cs, state_grads=True, flags=flags)
        g["y"], g["h_T"], _ = binding.prefill(x, params, h0=h0, conv_state_in=cs, flags=flags)
        torch.cuda.synchronize()
        err.append({k: _norm_error(to_np(g[k]), ref[k]) for k in ref})
    for k in ref:
        assert err[0][k] <= err[1][k] * (1.001 if g[k].dtype == torch.bfloat16 else 1.0), (k, err[0][k], err[1][k])


def test_split_backward_keeps_an_overflowed_gradient_non_finite():
    """An infinite dy must not come out as finite weight gradients: loss scaling looks for it there.  It stays in its own head."""
    import torch
    from paper_2402_19427_b200 import binding
    T, Dh, H = 40, 64, 2
    inp = synth.make_inputs(1, T, Dh * H, H, io="f32", seed=4, with_dy=True)
    params = binding.Params.from_numpy(inp["params"], "f32")
    dy = to_dev(inp["dy"])
    dy[0, 20, 3] = float("inf")
    g = binding.backward(to_dev(inp["x"]), params, dy)
    torch.cuda.synchronize()
    for k in ("W_a", "W_x"):
        assert not bool(torch.isfinite(g[k][0, 3]).any()), k
        assert bool(torch.isfinite(g[k][1]).all()), k


def test_split_products_leave_out_no_more_than_a_rounding():
    """One token, so that every dW[o][n] is one product dz[o] u[n], with dz the db of the same call and u = x (taps 1, 0, 0, 0) of values
    whose lower sixteen bits are all ones.  The plane products that are left out come to at most 2^-24 of it, the sum of the two
    accumulators is rounded once (2^-24), the small one five times at 2^-7 of the size."""
    import torch
    from paper_2402_19427_b200 import binding
    Dh, H = 128, 2
    inp = synth.make_inputs(1, 1, Dh * H, H, io="f32", seed=12, with_dy=True)
    p = inp["params"]
    p["conv_w"][:] = 0.0
    p["conv_w"][0] = 1.0
    p["conv_b"][:] = 0.0
    x = (inp["x"].view(np.uint32) | np.uint32(0xFFFF)).view(np.float32)
    g = binding.backward(to_dev(x), binding.Params.from_numpy(p, "f32"), to_dev(inp["dy"]))
    torch.cuda.synchronize()
    u = x.astype(np.float64).reshape(H, 1, Dh)
    for W, b in (("W_a", "b_a"), ("W_x", "b_x")):
        want = to_np(g[b]).reshape(H, Dh, 1) * u
        worst = (np.abs(to_np(g[W]) - want) / np.abs(want)).max()
        assert worst <= 2.0 ** -23 + 5 * 2.0 ** -31, (W, worst * 2.0 ** 24)


@pytest.mark.parametrize("io,B,T,Dh,H", [("f32", 2, 70, 96, 3), ("f32", 3, 770, 64, 4), ("bf16", 2, 70, 288, 3)])   # 32 and 64 tokens a block
@pytest.mark.parametrize("what", ["x", "two x", "zero weight", "W_a", "W_x"])
def test_split_products_do_not_lose_an_infinity(io, B, T, Dh, H, what):
    """An infinite input or weight in one head: a gate whose sum is infinite saturates, one whose sum is not defined (infinities of both
    signs, an infinity times zero) gives NaN, as on the CUDA cores; no gradient is finite that is not finite there, and the other heads
    and (for an input) sequences do not see it."""
    import torch
    from paper_2402_19427_b200 import binding
    D = Dh * H
    inp = synth.make_inputs(B, T, D, H, io=io, seed=18, with_dy=True, with_state=True, bias_scale=0.2)
    p = inp["params"]
    c0 = Dh + 5   # a channel of the second head
    p["conv_w"][0, c0], p["conv_w"][0, c0 + 9] = 0.5, 0.5
    if what in ("W_a", "W_x"):
        p[what][1, 7, 5] = np.inf if what == "W_a" else -np.inf
    else:
        inp["x"][1, 20, c0] = np.inf
        if what == "two x":
            inp["x"][1, 20, c0 + 9] = -np.inf
        if what == "zero weight":
            p["W_a"][1, :40, 5] = 0.0
    params = binding.Params.from_numpy(p, io)
    x, h0, cs, dy = to_dev(inp["x"], io), to_dev(inp["h0"]), to_dev(inp["conv_state"], io), to_dev(inp["dy"], io)
    got, want = [], []
    for flags, out in ((0, got), (1, want)):   # 1: RGLRU_FLAG_FORCE_GENERIC
        y, hT, _ = binding.prefill(x, params, h0=h0, conv_state_in=cs, flags=flags)
        out += [y, hT, binding.backward(x, params, dy, h0=h0, conv_state_in=cs, state_grads=True, flags=flags)]
    torch.cuda.synchronize()
    for a, b in zip(got[:2], want[:2]):
        ok = torch.isfinite(b)
        assert torch.equal(torch.isfinite(a), ok)
        assert what in ("W_a", "W_x") or bool((~ok).any())   # an infinite weight only saturates its gate
        np.testing.assert_allclose(to_np(a[ok]), to_np(b[ok]), rtol=2e-2 if io == "bf16" else 1e-4, atol=1e-3 if io == "bf16" else 1e-5)
    for k, b in want[2].items():
        a = got[2][k]
        assert not bool((torch.isfinite(a) & ~torch.isfinite(b)).any()), k
        per_head = a.view(H, -1) if k in ("W_a", "W_x") else a.view(-1, H, Dh).transpose(0, 1)
        assert bool(torch.isfinite(per_head[0]).all()) and bool(torch.isfinite(per_head[2]).all()), k
    if what not in ("W_a", "W_x"):
        assert bool(torch.isfinite(got[0][0]).all()) and bool(torch.isfinite(got[2]["x"][0]).all())


@pytest.mark.parametrize("B,T,Dh,H,few", [
    (1, 1, 128, 8, True), (1, 128, 256, 4, True), (1, 129, 256, 4, False), (1, 32, 256, 18, True), (1, 32, 256, 19, False),
    (37, 9, 32, 8, True), (38, 9, 32, 8, False), (1, 33, 1024, 2, True), (2, 33, 1024, 2, False)])
def test_fp32_forward_of_few_tokens_is_left_to_the_cuda_cores(oracle, B, T, Dh, H, few):
    """Both sides of the rule: the CUDA cores' own results, bit for bit, where they take the call, with a workspace as small as theirs;
    the call is right on either side, state in place."""
    import torch
    from paper_2402_19427_b200 import binding
    D = Dh * H
    inp = synth.make_inputs(B, T, D, H, io="f32", seed=400 + T, with_state=True, bias_scale=0.2)
    params = binding.Params.from_numpy(inp["params"], "f32")
    out, size = [], []
    for flags in (0, 1):   # 1: RGLRU_FLAG_FORCE_GENERIC
        h, c = to_dev(inp["h0"]), to_dev(inp["conv_state"])
        shape = binding.make_shape(B, T, D, H, torch.float32, flags=flags)
        size.append(binding.workspace_bytes(shape, binding.OP_PREFILL))
        y, _, _ = binding.prefill(to_dev(inp["x"]), params, h0=h, conv_state_in=c, h_T=h, conv_state_out=c, flags=flags)
        out.append((y, h, c))
    torch.cuda.synchronize()
    assert (size[0] == size[1]) == few
    assert torch.equal(out[0][0], out[1][0]) == few and torch.equal(out[0][2], out[1][2])
    yr, hr, cr = oracle_prefill(oracle, inp, h0=inp["h0"].astype(np.float64), cs=inp["conv_state"].astype(np.float64))
    assert_close("y", to_np(out[0][0]), yr, "f32"); assert_close("h_T", to_np(out[0][1]), hr, "f32")
    assert np.array_equal(to_np(out[0][2]), cr)


def test_host_prefill_whose_shares_cross_that_rule(oracle):
    """The whole batch is beyond the rule, the shares that the call cuts it into are not: a workspace for the whole serves them all."""
    import torch
    from paper_2402_19427_b200 import binding
    B, T, Dh, H = 6, 100, 128, 8
    inp = synth.make_inputs(B, T, Dh * H, H, io="f32", seed=7)
    D, params = Dh * H, binding.Params.from_numpy(inp["params"], "f32")
    y, hT, cs = [torch.empty(*s, pin_memory=True) for s in ((B, T, D), (B, D), (B, 3, D))]
    shape = binding.make_shape(B, T, D, H, torch.float32)
    staging = torch.empty(binding.host_staging_bytes(shape), dtype=torch.uint8, device="cuda")
    binding.prefill_host(torch.from_numpy(inp["x"]).pin_memory(), params, y, hT, cs, staging, binding.alloc_workspace(shape, binding.OP_PREFILL, staging.device))
    torch.cuda.synchronize()
    yr, hr, cr = oracle_prefill(oracle, inp)
    assert_close("y", to_np(y), yr, "f32"); assert_close("h_T", to_np(hT), hr, "f32")
    assert np.array_equal(to_np(cs), cr)


def test_backward_in_passes_over_the_sequences():
    """A call whose arrays would take more than 4 GiB goes through its sequences in passes, three of two sequences at most here.  What
    belongs to a sequence is bit for bit what a call of its pass alone gives, what is summed over them is the sum (in another order: 2^-22)."""
    import torch
    from paper_2402_19427_b200 import binding
    B, T, D, H = 5, 8203, 4096, 32
    assert binding.workspace_bytes(binding.make_shape(B, T, D, H, torch.bfloat16), binding.OP_BACKWARD) < 20 * B * T * D
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    params = binding.Params.from_numpy(synth.make_inputs(1, 1, D, H, io="bf16", seed=6, bias_scale=0.2)["params"], "bf16")
    f32 = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    bf16 = lambda *s: f32(*s).to(torch.bfloat16)
    x, dy, h0, cs, dhT, dcs = bf16(B, T, D), bf16(B, T, D), f32(B, D), bf16(B, 3, D), f32(B, D), bf16(B, 3, D)
    call = lambda s: binding.backward(x[s], params, dy[s], h0=h0[s], conv_state_in=cs[s], dh_T=dhT[s], dconv_state_out=dcs[s], state_grads=True)
    whole, parts = call(slice(0, 5)), [call(slice(0, 2)), call(slice(2, 4)), call(slice(4, 5))]
    torch.cuda.synchronize()
    for k, v in whole.items():
        if k in ("x", "h0", "conv_state"):
            assert torch.equal(v, torch.cat([g[k] for g in parts])), k
        else:
            want = sum(g[k].double() for g in parts)
            assert float((v.double() - want).norm() / want.norm()) < 2.0 ** -22, k


def test_gates_of_the_split_forward_are_good_to_their_last_places():
    """Zero gate weights, so that r and i are the sigmoids of the biases, and an impulse: y_0 = m i u, y_1 = a y_0, for every channel another
    r, i and decay.  i, m and the decay rate are within 2 units in the last place (4 x 2^-24), the error of r and of the rate enters m by
    half (4), and there are two products (2): 14 x 2^-24 for y_0, and as much again for a, which is 1/2 at least."""
    import torch
    from paper_2402_19427_b200 import binding
    T, Dh, H = 160, 256, 16
    D = Dh * H
    p = synth.make_inputs(1, 1, D, H, io="f32", seed=2)["params"]
    rng = np.random.default_rng(8)
    for k in ("W_a", "W_x", "conv_w", "conv_b"):
        p[k][:] = 0.0
    p["conv_w"][0] = 1.0
    p["b_a"][:], p["b_x"][:] = rng.uniform(-12, 12, D), rng.uniform(-12, 12, D)
    a_c = np.where(rng.random(D) < 0.5, rng.uniform(0.5, 0.999, D), 1.0 - 10.0 ** rng.uniform(-6, -3, D))
    p["lam"][:] = np.log(a_c ** 0.125 / (1.0 - a_c ** 0.125))
    x = torch.zeros(1, T, D, device="cuda")
    x[0, 0] = torch.from_numpy(rng.standard_normal(D)).float()
    y = to_np(binding.prefill(x, binding.Params.from_numpy(p, "f32"))[0])[0]
    b_a, b_x, lam, u = p["b_a"].astype(np.float64), p["b_x"].astype(np.float64), p["lam"].astype(np.float64), to_np(x)[0, 0]
    L = 8.0 * np.log1p(np.exp(-lam)) / (1.0 + np.exp(-b_a))
    y0 = np.sqrt(-np.expm1(-2.0 * L)) * u / (1.0 + np.exp(-b_x))
    assert (np.abs(y[0] - y0) / np.abs(y0)).max() <= 14 * 2.0 ** -24
    assert (np.abs(y[1] - np.exp(-L) * y0) / np.abs(np.exp(-L) * y0)).max() <= 28 * 2.0 ** -24
