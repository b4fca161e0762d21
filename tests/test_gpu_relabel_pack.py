"""The update step's relabel, which writes the BF16 network inputs itself, against
sampling and a critic step on the sampled batch: the same indices and the same split
inputs give the same critic loss and gradients, bit for bit."""

import pytest
import torch

from parity_helpers import setup, small

pytestmark = pytest.mark.gpu


# batches around the 16 samples of a block; widths off a warp's 32 columns; every goal dim
@pytest.mark.parametrize("B,D,A,G", [(8, 3, 1, 1), (24, 29, 8, 2), (136, 33, 17, 16), (256, 268, 17, 3)])
def test_update_step_inputs_equal_sampled_ones(B, D, A, G):
    w = small(B=B, D=D, A=A, G=min(G, D), hidden=64, layers=1, repr=64)
    one, two = (setup(w, precision="bf16", path="fused")[0] for _ in range(2))
    loss = torch.zeros(6, device="cuda")
    parts = torch.zeros(4, device="cuda")
    step = one.get_step()
    one.update_step(loss_out=loss)
    s, a, g, _ = two.sample(step)
    two.critic_step(s, a, g, loss_out=parts)
    torch.cuda.synchronize()
    assert torch.equal(loss[:4], parts)
    for net in ("phi", "psi"):
        assert torch.equal(one.store[net]["grads"], two.store[net]["grads"])
