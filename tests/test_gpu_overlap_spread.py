"""Launch overlap does not crowd the FP32 products and the -L1 gradients onto part of
the SMs: the plain loss backward takes no longer with overlapping launches than
without.  (Crowded, the sizes here took 1.3 to 1.7 times as long.)"""

from ctypes import byref, c_size_t

import pytest
import torch

from paper_2408_11052_gb300 import api

pytestmark = pytest.mark.gpu


def backward_us(prec, B, R, energy, loss):
    L, st = api.lib(), api.stream_handle()
    dt = torch.float64 if prec == "fp64" else torch.float32
    desc = api.CrlLossDesc(api.ENERGY[energy], api.LOSS[loss], api.SYM["mean"], api.PENALTY["row"], 1.0, 0.1,
                           api.PREC[prec], api.PATH["plain"])
    g = torch.Generator(device="cuda").manual_seed(9)
    phi, psi = (torch.randn(B, R, device="cuda", dtype=dt, generator=g) for _ in range(2))
    dphi, dpsi, n = torch.empty_like(phi), torch.empty_like(psi), c_size_t()
    api.check(L.crl_infonce_workspace_bytes(byref(desc), B, R, byref(n)))
    ws = torch.empty(n.value, dtype=torch.uint8, device="cuda")
    parts, r, c = torch.empty(4, device="cuda", dtype=dt), phi[:, 0].clone(), phi[:, 0].clone()
    api.check(L.crl_infonce_forward(byref(desc), phi.data_ptr(), psi.data_ptr(), B, R, parts.data_ptr(), r.data_ptr(),
                                    c.data_ptr(), ws.data_ptr(), n.value, st))
    best = {}
    for _ in range(8):                            # (the two settings in turn)
        for on in (True, False):
            prev = api.set_launch_overlap(on)
            try:
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                torch.cuda._sleep(1_000_000)      # the launches queue up: device time only
                a.record()
                for _ in range(6):
                    api.check(L.crl_infonce_backward(byref(desc), phi.data_ptr(), psi.data_ptr(), B, R, r.data_ptr(),
                                                     c.data_ptr(), 1.0, dphi.data_ptr(), dpsi.data_ptr(),
                                                     ws.data_ptr(), n.value, st))
                b.record()
                torch.cuda.synchronize()
            finally:
                api.set_launch_overlap(prev)
            best[on] = min(best.get(on, float("inf")), a.elapsed_time(b) / 6e-3)
    return best[True], best[False]


@pytest.mark.parametrize("prec,B,R,energy,loss", [
    ("fp32", 1001, 200, "l1", "sym"), ("fp64", 512, 64, "l1", "sym"), ("fp32", 2048, 64, "cos", "fwd")])
def test_overlapping_launches_are_spread(prec, B, R, energy, loss):
    overlapped, apart = backward_us(prec, B, R, energy, loss)
    assert overlapped < 1.1 * apart, (overlapped, apart)
