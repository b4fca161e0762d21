"""Op-level BF16 encoder calls whose output and gradient arrays start on a 4-byte
boundary (the entry points ask for no more): the same bits as in aligned arrays, and
nothing outside the rows.  Widths below and above one 32-column step, an output of a
whole wide tile, and a batch whose weight gradients are split over K."""

from ctypes import byref, c_size_t

import pytest
import torch

from paper_2408_11052_gb300 import api

pytestmark = pytest.mark.gpu

GUARD = 7.5


def at_offset(n, off):
    """n floats that start `off` floats past a 256-byte boundary, and the array they stand in."""
    whole = torch.full((n + 128,), GUARD, device="cuda")
    return whole[64 + off:64 + off + n], whole


@pytest.mark.parametrize("M,hidden,layers,out,layernorm", [
    (40, 8, 1, 8, 0), (40, 16, 2, 16, 0), (129, 24, 2, 12, 1), (33, 64, 1, 64, 0), (257, 72, 2, 20, 0),
    (8192, 64, 2, 64, 0), (4096, 256, 1, 256, 0),
])
def test_outputs_on_four_byte_boundaries(M, hidden, layers, out, layernorm):
    g = torch.Generator(device="cuda").manual_seed(6)
    in0 = 29
    desc = api.CrlMlpDesc(in0, 0, hidden, layers, out, layernorm, api.PREC["bf16"])
    up = lambda n: -(-n // 64) * 64
    dims = [in0] + [hidden] * layers + [out]
    n = sum(up(a * b) + up(b) for a, b in zip(dims, dims[1:])) + (2 * layers * up(hidden) if layernorm else 0)
    params = 0.1 * torch.randn(n, device="cuda", generator=g)
    x0 = torch.randn(M, in0, device="cuda", generator=g)
    dy0 = torch.randn(M, out, device="cuda", generator=g)
    L, nb, st = api.lib(), c_size_t(), api.stream_handle()
    api.check(L.crl_mlp_saved_bytes(byref(desc), M, byref(nb)))
    got = []
    for off in (0, 1, 2):
        saved = torch.empty(nb.value, dtype=torch.uint8, device="cuda")
        (y, yw), (dp, dpw), (dx, dxw), (dy, _) = (at_offset(k, off) for k in (M * out, n, M * in0, M * out))
        dy.copy_(dy0.reshape(-1))
        api.check(L.crl_mlp_forward(byref(desc), params.data_ptr(), x0.data_ptr(), None, M, y.data_ptr(),
                                    saved.data_ptr(), st))
        api.check(L.crl_mlp_backward(byref(desc), params.data_ptr(), x0.data_ptr(), None, M, saved.data_ptr(),
                                     dy.data_ptr(), dp.data_ptr(), dx.data_ptr(), None, st))
        torch.cuda.synchronize()
        for whole in (yw, dpw, dxw):
            assert (whole[:64 + off] == GUARD).all() and (whole[len(whole) - 64 + off:] == GUARD).all()
        got.append((y, dp, dx))
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert torch.equal(a, b)
