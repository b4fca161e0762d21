"""The critic's two encoders share their launches in the FP32 / FP64 critic step: the
gradients equal, bit for bit, those of the encoders run one after the other through
the op-level calls (every output is one sum in a fixed order, whatever the tile)."""

import numpy as np
import pytest
import torch

from paper_2408_11052_gb300 import api, functional, workload

from parity_helpers import small

pytestmark = pytest.mark.gpu


# networks of unlike input widths; batches and widths off every tile; one layer to three
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("B,D,A,G,hidden,layers,layernorm", [
    (1, 3, 1, 1, 8, 1, False), (33, 29, 8, 2, 68, 2, True), (96, 120, 20, 8, 80, 3, True), (256, 29, 8, 2, 256, 2, False),
])
def test_pair_equals_one_by_one(B, D, A, G, hidden, layers, layernorm, precision):
    w = small(B=B, D=D, A=A, G=G, hidden=hidden, layers=layers, layernorm=layernorm)
    ctx = api.CRLContext(w, precision=precision, path="plain")
    for k, v in workload.init_agent(w, perturb=True).items():
        ctx.load_network(k, v)
    g = torch.Generator(device="cuda").manual_seed(2)
    s, a, goal = (torch.randn(B, n, device="cuda", generator=g) for n in (D, A, G))
    ctx.critic_step(s, a, goal)
    pp = ctx.store["phi"]["params"].clone().requires_grad_(True)
    pq = ctx.store["psi"]["params"].clone().requires_grad_(True)
    phi = functional.encoder(pp, s, a, D, A, hidden, layers, w.repr, layernorm)
    psi = functional.encoder(pq, goal, None, G, 0, hidden, layers, w.repr, layernorm)
    total, _ = functional.infonce_loss(phi, psi, w.energy, w.loss, w.sym_reduction, w.penalty_axis,
                                       float(np.float32(w.tau)), float(np.float32(w.beta)), "plain")
    total.backward()
    torch.cuda.synchronize()
    assert torch.equal(ctx.store["phi"]["grads"], pp.grad)
    assert torch.equal(ctx.store["psi"]["grads"], pq.grad)
