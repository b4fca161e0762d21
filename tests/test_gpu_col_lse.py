"""The plain path's row and column logsumexps where their blocks end: batches around the
32 columns and the 32 x 8 rows of a step, in FP32 and FP64, against torch.logsumexp in
FP64 of the energy matrix itself (dot products of the same representations)."""

from ctypes import byref, c_size_t

import pytest
import torch

from paper_2408_11052_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("B", [1, 2, 31, 33, 64, 255, 257, 545])
def test_logsumexps(prec, B):
    R, L = 24, api.lib()
    dt = torch.float64 if prec == "fp64" else torch.float32
    desc = api.CrlLossDesc(api.ENERGY["dot"], api.LOSS["sym"], api.SYM["mean"], api.PENALTY["row"], 1.0, 0.1,
                           api.PREC[prec], api.PATH["plain"])
    g = torch.Generator(device="cuda").manual_seed(B)
    phi, psi = (2.0 * torch.randn(B, R, device="cuda", dtype=dt, generator=g) for _ in range(2))
    n = c_size_t()
    api.check(L.crl_infonce_workspace_bytes(byref(desc), B, R, byref(n)))
    ws = torch.empty(n.value, dtype=torch.uint8, device="cuda")
    parts, r, c = (torch.empty(k, device="cuda", dtype=dt) for k in (4, B, B))
    api.check(L.crl_infonce_forward(byref(desc), phi.data_ptr(), psi.data_ptr(), B, R, parts.data_ptr(), r.data_ptr(),
                                    c.data_ptr(), ws.data_ptr(), n.value, api.stream_handle()))
    F = phi.double() @ psi.double().T
    # a sum of 24 products of this type and a logarithm: |F| terms of relative rounding each
    scale = (phi.double().abs() @ psi.double().abs().T).max().item() + 10.0
    tol = 32 * torch.finfo(dt).eps * scale
    for got, dim in ((r, 1), (c, 0)):
        want = torch.logsumexp(F, dim=dim)
        assert (got.double() - want).abs().max().item() <= tol
