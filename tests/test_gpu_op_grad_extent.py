"""Where the BF16 encoder backward writes in the caller's gradient array: the whole
layout, every tensor's padding included, and nothing after it.  The autograd wrapper
takes parameters that end with the last bias as well (its own array then holds the
rest of the layout); its gradient's padding is zero."""

from ctypes import byref, c_size_t

import pytest
import torch

from paper_2408_11052_gb300 import api, functional


class Recorder:
    """In the compiled library's place: keeps the call's arguments."""

    def crl_mlp_backward(self, *args):
        self.args = args
        return 0


@pytest.mark.parametrize("extra", [-45, 0, 9])
def test_the_wrapper_hands_over_the_whole_layout(monkeypatch, extra):
    """CPU: the array that the BF16 backward writes holds the layout whatever the parameters' length."""
    desc, _, count = functional._mlp_plan(5, 0, 40, 1, 19, 0, api.PREC["bf16"], 3)
    params = torch.zeros(count + extra)            # out = 19: 45 elements of padding end the layout

    class Ctx:
        saved_tensors = params, torch.zeros(3, 5), None, torch.zeros(8, dtype=torch.uint8)
        has_x1, needs_input_grad = False, (True, False, False)

    ctx, lib = Ctx(), Recorder()
    ctx.desc, ctx.count = desc, count
    monkeypatch.setattr(api, "lib", lambda: lib)
    monkeypatch.setattr(api, "stream_handle", lambda *a: 0)
    grad = functional.EncoderMLP.backward(ctx, torch.zeros(3, 19))[0]
    assert grad.shape == params.shape and lib.args[7] == grad.data_ptr()
    assert grad.untyped_storage().nbytes() // 4 >= count


@pytest.mark.gpu
@pytest.mark.parametrize("M,in0,hidden,layers,out,layernorm", [
    (33, 5, 40, 1, 19, 0), (40, 3, 16, 2, 8, 1), (129, 29, 64, 2, 64, 0), (8192, 29, 64, 2, 72, 0)])
def test_the_gradient_array_ends_with_the_layout(M, in0, hidden, layers, out, layernorm):
    g = torch.Generator(device="cuda").manual_seed(7)
    desc = api.CrlMlpDesc(in0, 0, hidden, layers, out, layernorm, api.PREC["bf16"])
    up = lambda n: -(-n // 64) * 64
    dims = [in0] + [hidden] * layers + [out]
    n = sum(up(a * b) + up(b) for a, b in zip(dims, dims[1:])) + (2 * layers * up(hidden) if layernorm else 0)
    end = n - up(out) + out                      # one past the last bias
    params = 0.1 * torch.randn(n, device="cuda", generator=g)
    x0 = torch.randn(M, in0, device="cuda", generator=g)
    dy = torch.randn(M, out, device="cuda", generator=g)
    L, nb, st = api.lib(), c_size_t(), api.stream_handle()
    api.check(L.crl_mlp_saved_bytes(byref(desc), M, byref(nb)))
    saved = torch.empty(nb.value, dtype=torch.uint8, device="cuda")
    y, dp = torch.empty(M, out, device="cuda"), torch.full((n + 64,), float("nan"), device="cuda")
    api.check(L.crl_mlp_forward(byref(desc), params.data_ptr(), x0.data_ptr(), None, M, y.data_ptr(),
                                saved.data_ptr(), st))
    api.check(L.crl_mlp_backward(byref(desc), params.data_ptr(), x0.data_ptr(), None, M, saved.data_ptr(),
                                 dy.data_ptr(), dp.data_ptr(), None, None, st))
    torch.cuda.synchronize()
    assert torch.isfinite(dp[:end]).all() and (dp[end:n] == 0).all() and torch.isnan(dp[n:]).all()

    def grad(p):
        p = p.clone().requires_grad_(True)
        return torch.autograd.grad(functional.encoder(p, x0, None, in0, 0, hidden, layers, out, layernorm, "bf16"),
                                   p, dy)[0]

    whole = grad(params)
    assert torch.equal(whole, dp[:n])
    short = grad(params[:end])                   # parameters that end with the last bias
    assert short.shape == (end,) and torch.equal(short, dp[:end])
    longer = grad(torch.cat([params, params[:9]]))
    assert torch.equal(longer[:n], dp[:n]) and (longer[n:] == 0).all()
