"""The autograd wrappers keep descriptors per value: options may be anything that
converts to a number (0-d tensors and arrays, NumPy scalars), are read on every call,
and are refused where they do not convert."""

import numpy as np
import pytest
import torch

from paper_2408_11052_gb300 import api, functional


def loss_plan(temperature, beta):
    return functional._loss_plan("l2", "sym", "mean", "row", temperature, beta, api.PREC["fp32"], "plain", 24, 16)[0]


def mlp_plan(in0, hidden):
    return functional._mlp_plan(in0, 2, hidden, 1, 8, 0, api.PREC["fp32"], 24)


def test_loss_options_are_read_on_every_call():
    for make in (torch.tensor, np.array):
        tau, beta = make(1.0), make(0.25)
        first = loss_plan(tau, beta)
        assert (first.temperature, first.beta_lse) == (1.0, 0.25)
        tau *= 0.5
        beta *= 2.0
        second = loss_plan(tau, beta)
        assert (second.temperature, second.beta_lse) == (0.5, 0.5)
        assert (first.temperature, first.beta_lse) == (1.0, 0.25)   # a graph that was recorded keeps its own
    assert loss_plan(np.float32(2), 1).temperature == 2.0
    for bad in ("1.0", None):
        with pytest.raises(TypeError):
            loss_plan(bad, 0.1)


def test_widths_are_read_on_every_call():
    for make in (torch.tensor, np.array):
        in0, hidden = make(3), make(16)
        _, nbytes, count = mlp_plan(in0, hidden)
        assert count == mlp_plan(3, 16)[2] == 128 + 64 + 128 + 64
        in0 += 61
        hidden += 16
        desc, wider, wide = mlp_plan(in0, hidden)
        assert (desc.in0, desc.hidden) == (64, 32) and wider > nbytes
        assert wide == mlp_plan(64, np.int64(32))[2]
    with pytest.raises(TypeError):
        mlp_plan(3.0, 16)


@pytest.mark.gpu
@pytest.mark.parametrize("path", ["plain", "fused"])
def test_a_changed_temperature_tensor_changes_the_loss(path):
    g = torch.Generator(device="cuda").manual_seed(8)
    phi, psi = (torch.randn(24, 64, device="cuda", generator=g) for _ in range(2))
    tau = torch.tensor(1.0)
    functional.infonce_loss(phi, psi, temperature=tau, path=path)
    tau.mul_(0.5)
    got = functional.infonce_loss(phi, psi, temperature=tau, beta=np.array(0.1), path=path)
    want = functional.infonce_loss(phi, psi, temperature=0.5, beta=0.1, path=path)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
