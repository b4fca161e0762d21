"""The BF16 critic step refreshes each encoder's weight shadows in one launch, and the
shadows are those of any other call: the same losses and gradients from the FP32
masters at depths and widths off the 64 x 64 weight tiles."""

import pytest
import torch

from paper_2408_11052_gb300 import api, workload

from parity_helpers import small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,layers,B", [(256, 2, 64), (72, 1, 8), (104, 5, 40)])
def test_one_shadow_launch_per_network(hidden, layers, B):
    w = small(B=B, hidden=hidden, layers=layers, repr=64)
    ctx = api.CRLContext(w, precision="bf16", path="fused")
    for k, v in workload.init_agent(w, perturb=True).items():
        ctx.load_network(k, v)
    obs, act, done = workload.buffer_contents(w, mean_len=9.0)
    ctx.insert(*(torch.from_numpy(x).to(ctx.device) for x in (obs, act, done)))
    s, a, g, _ = ctx.sample(3)
    first = ctx.critic_step(s, a, g).clone()
    grads = [ctx.store[n]["grads"].clone() for n in ("phi", "psi")]
    ctx.trace_start("aux", 64)
    again = ctx.critic_step(s, a, g)
    assert ctx.trace_stop()[0] == 4          # phi and psi: shadows, input
    torch.cuda.synchronize()
    assert torch.equal(first, again)
    for before, n in zip(grads, ("phi", "psi")):
        assert torch.equal(before, ctx.store[n]["grads"])
