"""Collection in one launch (FP32 policies that fit in shared memory) against the
layer-by-layer path, bit for bit, at its edges: environments and columns that do not
fill their tiles, every cluster size, one to three layers, LayerNorm, episodes that
end inside a call, more steps than one launch takes.  An environment's draws and
arithmetic do not depend on how many others there are, and a batch too large for the
one launch takes the layers one by one."""

import numpy as np
import pytest
import torch

from paper_2408_11052_gb300 import api, workload

from parity_helpers import small

MANY = 40000   # more environments than the one launch takes at any size

pytestmark = pytest.mark.gpu


def collect(w, n, L, calls=1):
    ctx = api.CRLContext(w, precision="fp32", path="plain")
    nets = workload.init_agent(w, perturb=True)
    for k, v in nets.items():
        ctx.load_network(k, v)
    out = [(torch.zeros(n, w.E, w.D, device=ctx.device), torch.zeros(n, w.E, w.A, device=ctx.device),
            torch.zeros(n, w.E, dtype=torch.uint8, device=ctx.device)) for _ in range(calls)]
    for o in out:
        ctx.collect(n, L, out=o)
    torch.cuda.synchronize()
    return ctx, [np.concatenate([o[i].cpu().numpy() for o in out]) for i in range(3)]


@pytest.mark.parametrize("E,D,A,G,hidden,layers,layernorm", [
    (1, 3, 1, 1, 4, 1, False),         # one CTA, one tile
    (37, 30, 7, 3, 68, 1, True),       # ragged environments, columns and noise pairs
    (130, 29, 8, 2, 256, 2, False),    # two CTAs per cluster
    (1024, 29, 8, 2, 256, 2, True),
    (70, 200, 17, 9, 256, 2, True),    # a wide input: more CTAs per cluster
    (33, 12, 5, 3, 204, 3, False),
    (40, 20, 6, 2, 512, 2, False),     # eight CTAs
])
def test_unroll_matches_the_layer_path(E, D, A, G, hidden, layers, layernorm):
    n, L = 19, 6                       # the ring wraps; episodes end inside the call
    few, many = (small(E=e, T=16, B=16, D=D, A=A, G=G, hidden=hidden, layers=layers,
                       layernorm=layernorm) for e in (E, MANY))
    ctx, got = collect(few, n, L)
    assert ctx.buffer_size() == (few.T, n)
    _, want = collect(many, n, L)
    for a, b in zip(got, want):
        assert np.isfinite(a).all()
        np.testing.assert_array_equal(a, b[:, :E])


def test_more_steps_than_one_launch_takes():
    w = small(E=4, T=64, B=16)
    _, one = collect(w, 1040, 50)
    _, many = collect(w, 208, 50, calls=5)
    for a, b in zip(one, many):
        np.testing.assert_array_equal(a, b)
