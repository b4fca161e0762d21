"""The op-level BF16 calls on workspaces that held anything, and the InfoNCE
backward with its multiplier in device memory.  Every result is compared bit for
bit: with the same call on a cleared workspace, and with the host multiplier."""

from ctypes import byref, c_size_t

import pytest
import torch

from paper_2408_11052_gb300 import api, functional

pytestmark = pytest.mark.gpu


def _mlp(desc, M, params, x0, x1, dy, fill):
    L = api.lib()
    n = c_size_t()
    api.check(L.crl_mlp_saved_bytes(byref(desc), M, byref(n)))
    saved = torch.full((n.value,), fill, dtype=torch.uint8, device="cuda")
    y = torch.empty(M, desc.out, device="cuda")
    dp = torch.full_like(params, float("nan"))
    dx = [torch.empty_like(x0), None if x1 is None else torch.empty_like(x1)]
    st = api.stream_handle()
    api.check(L.crl_mlp_forward(byref(desc), params.data_ptr(), x0.data_ptr(), api.ptr(x1), M, y.data_ptr(),
                                saved.data_ptr(), st))
    api.check(L.crl_mlp_backward(byref(desc), params.data_ptr(), x0.data_ptr(), api.ptr(x1), M, saved.data_ptr(),
                                 dy.data_ptr(), dp.data_ptr(), dx[0].data_ptr(), api.ptr(dx[1]), st))
    torch.cuda.synchronize()
    return [t for t in (y, dp, *dx) if t is not None]


# hidden and input widths off the 64-column padding and off the 64 x 64 weight
# tiles, odd row counts, one wide and one deep network, a batch that splits K
@pytest.mark.parametrize("M,in0,in1,hidden,layers,out,layernorm", [
    (1, 3, 0, 8, 1, 8, 0),
    (33, 5, 2, 40, 1, 19, 0),           # an output width off the 16-byte pitch
    (129, 29, 8, 72, 2, 64, 1),
    (257, 61, 3, 200, 3, 72, 1),
    (1000, 268, 17, 256, 4, 64, 0),
    (8192, 64, 16, 64, 2, 64, 0),
])
def test_encoder_on_a_dirty_workspace(M, in0, in1, hidden, layers, out, layernorm):
    g = torch.Generator(device="cuda").manual_seed(3)
    desc = api.CrlMlpDesc(in0, in1, hidden, layers, out, layernorm, api.PREC["bf16"])
    up = lambda n: -(-n // 64) * 64
    dims = [in0 + in1] + [hidden] * layers + [out]
    n = sum(up(a * b) + up(b) for a, b in zip(dims, dims[1:])) + (2 * layers * up(hidden) if layernorm else 0)
    params = 0.1 * torch.randn(n, device="cuda", generator=g)
    x0 = torch.randn(M, in0, device="cuda", generator=g)
    x1 = torch.randn(M, in1, device="cuda", generator=g) if in1 else None
    dy = torch.randn(M, out, device="cuda", generator=g)
    clean = _mlp(desc, M, params, x0, x1, dy, 0)
    dirty = _mlp(desc, M, params, x0, x1, dy, 0xFF)   # NaN in every type
    for a, b in zip(clean, dirty):
        assert torch.isfinite(a).all()
        assert torch.equal(a, b)


@pytest.mark.parametrize("energy", ["l2", "cos", "l1"])
@pytest.mark.parametrize("B,R", [(8, 64), (264, 192), (520, 256)])
def test_infonce_on_a_dirty_workspace(B, R, energy):
    g = torch.Generator(device="cuda").manual_seed(4)
    phi = torch.randn(B, R, device="cuda", generator=g)
    psi = torch.randn(B, R, device="cuda", generator=g)
    L = api.lib()
    desc = api.CrlLossDesc(api.ENERGY[energy], api.LOSS["sym"], api.SYM["mean"], api.PENALTY["row"], 1.0, 0.1,
                           api.PREC["bf16"], api.PATH["fused"])
    n = c_size_t()
    api.check(L.crl_infonce_workspace_bytes(byref(desc), B, R, byref(n)))
    got = []
    for fill in (0, 0xFF):
        ws = torch.full((n.value,), fill, dtype=torch.uint8, device="cuda")
        parts, total = torch.empty(4, device="cuda"), torch.empty(1, device="cuda")
        r, c = torch.empty(B, device="cuda"), torch.empty(B, device="cuda")
        api.check(L.crl_infonce_forward_total(byref(desc), phi.data_ptr(), psi.data_ptr(), B, R, parts.data_ptr(),
                                              total.data_ptr(), r.data_ptr(), c.data_ptr(), ws.data_ptr(), n.value,
                                              api.stream_handle()))
        got.append((total, parts, r, c))
    for a, b in zip(*got):
        assert torch.equal(a, b)
    assert torch.equal(got[0][0], got[0][1][:1])


@pytest.mark.parametrize("path,dtype,energy,loss", [
    ("fused", torch.float32, "l2", "sym"), ("fused", torch.float32, "l1", "sym"),
    ("fused", torch.float32, "dot", "fb"), ("plain", torch.float32, "l2", "fwd"),
    ("plain", torch.float32, "cos", "nce_binary"), ("plain", torch.float64, "l2", "sym"),
])
def test_device_multiplier_equals_the_host_one(path, dtype, energy, loss):
    B, R, scale = 136, 64, 0.7
    g = torch.Generator(device="cuda").manual_seed(5)
    phi = torch.randn(B, R, device="cuda", dtype=dtype, generator=g).requires_grad_(True)
    psi = torch.randn(B, R, device="cuda", dtype=dtype, generator=g).requires_grad_(True)
    total, parts = functional.infonce_loss(phi, psi, energy=energy, loss=loss, path=path)
    k = torch.full((), scale, dtype=dtype, device="cuda")
    dphi, dpsi = torch.autograd.grad(total, (phi, psi), k)
    code = "bf16" if path == "fused" else {torch.float32: "fp32", torch.float64: "fp64"}[dtype]
    desc = api.CrlLossDesc(api.ENERGY[energy], api.LOSS[loss], api.SYM["mean"], api.PENALTY["row"], 1.0, 0.1,
                           api.PREC[code], api.PATH[path])
    L, n = api.lib(), c_size_t()
    api.check(L.crl_infonce_workspace_bytes(byref(desc), B, R, byref(n)))
    ws = torch.empty(n.value, dtype=torch.uint8, device="cuda")
    host = [torch.empty_like(t) for t in (parts, phi[:, 0], phi[:, 0], phi, phi)]
    p, r, c, a, b = (t.detach() for t in host)
    st = api.stream_handle()
    api.check(L.crl_infonce_forward(byref(desc), phi.data_ptr(), psi.data_ptr(), B, R, p.data_ptr(), r.data_ptr(),
                                    c.data_ptr(), ws.data_ptr(), n.value, st))
    api.check(L.crl_infonce_backward(byref(desc), phi.data_ptr(), psi.data_ptr(), B, R, r.data_ptr(), c.data_ptr(),
                                     k.item(), a.data_ptr(), b.data_ptr(), ws.data_ptr(), n.value, st))
    torch.cuda.synchronize()
    assert torch.equal(parts, p) and torch.equal(total.detach(), p[0])
    assert torch.equal(dphi, a) and torch.equal(dpsi, b)
