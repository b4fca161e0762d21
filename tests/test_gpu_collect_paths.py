"""Which path a collection call takes, seen in its launches (one product launch for the
one-launch path, one per layer and step for the layers), and that the paths may
alternate on one context: short calls of many environments are the layers', whose
bits a long call in one launch repeats."""

import numpy as np
import pytest
import torch

from paper_2408_11052_gb300 import api, workload

from parity_helpers import small

pytestmark = pytest.mark.gpu


def context(w):
    ctx = api.CRLContext(w, precision="fp32", path="plain")
    for k, v in workload.init_agent(w, perturb=True).items():
        ctx.load_network(k, v)
    return ctx


def product_launches(ctx, n, out=None):
    ctx.trace_start("gemm", 4096)
    ctx.collect(n, 6, out=out)
    return ctx.trace_stop()[0]


# the sizes of test_gpu_collect_unroll.py, whose few environments are to take the one launch
@pytest.mark.parametrize("E,D,A,G,hidden,layers,layernorm", [
    (1, 3, 1, 1, 4, 1, False), (37, 30, 7, 3, 68, 1, True), (130, 29, 8, 2, 256, 2, False),
    (1024, 29, 8, 2, 256, 2, True), (70, 200, 17, 9, 256, 2, True), (33, 12, 5, 3, 204, 3, False),
    (40, 20, 6, 2, 512, 2, False)])
def test_long_calls_take_one_launch(E, D, A, G, hidden, layers, layernorm):
    ctx = context(small(E=E, T=16, B=16, D=D, A=A, G=G, hidden=hidden, layers=layers, layernorm=layernorm))
    assert product_launches(ctx, 19) == 1
    many = context(small(E=40000, T=16, B=16, D=D, A=A, G=G, hidden=hidden, layers=layers, layernorm=layernorm))
    assert product_launches(many, 2) == 2 * (layers + 1)


@pytest.mark.parametrize("E,hidden,layers,layernorm,D", [
    (8192, 256, 2, False, 29), (4096, 256, 2, True, 268), (1024, 256, 3, False, 29)])
def test_one_step_of_many_environments_takes_the_layers(E, hidden, layers, layernorm, D):
    ctx = context(small(E=E, T=16, B=16, D=D, hidden=hidden, layers=layers, layernorm=layernorm))
    assert product_launches(ctx, 1) == layers + 1


@pytest.mark.parametrize("E,hidden,layernorm", [(64, 64, False), (1024, 256, False), (300, 128, True), (8192, 256, False)])
def test_calls_of_any_length_give_the_same_slices(E, hidden, layernorm):
    """31 steps as one call and as calls of 1, 2, 1, 3, 8 and 16 (episodes of 6 steps, a ring of 16)."""
    w = small(E=E, T=16, B=16, hidden=hidden, layers=2, layernorm=layernorm)
    got, paths = [], set()
    for parts in ((31,), (1, 2, 1, 3, 8, 16)):
        ctx, pieces = context(w), []
        for n in parts:
            out = (torch.zeros(n, w.E, w.D, device=ctx.device), torch.zeros(n, w.E, w.A, device=ctx.device),
                   torch.zeros(n, w.E, dtype=torch.uint8, device=ctx.device))
            paths.add(product_launches(ctx, n, out) == 1)
            pieces.append(out)
        torch.cuda.synchronize()
        got.append([np.concatenate([p[i].cpu().numpy() for p in pieces]) for i in range(3)] +
                   [np.frombuffer(ctx.save_state(), dtype=np.uint8)])
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
    if E == 8192:
        assert paths == {True, False}      # (both took part)
