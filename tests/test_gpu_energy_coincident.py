"""Fused -L2 backward where pairs coincide: d = 0 has coefficient 0 (the subgradient
rule), in interior tiles too, where the coefficient loop tests a whole group of
columns for coincident pairs at once.  Small integers are exact in BF16 and their
products in FP32, so d^2 of a coincident pair is exactly 0."""

import numpy as np
import pytest
import torch

import oracle
from paper_2408_11052_gb300 import functional

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("loss", ["fwd", "bwd", "sym"])
@pytest.mark.parametrize("B", [264, 512])
def test_coincident_pairs_off_the_diagonal(B, loss):
    rng = np.random.default_rng(5)
    phi = rng.integers(-2, 3, size=(B, 64)).astype(np.float32)
    psi = rng.integers(-2, 3, size=(B, 64)).astype(np.float32)
    # pairs in interior tiles, at a group's first and last column, and on the diagonal
    for i, j in ((3, 128), (7, 143), (130, 0), (200, 255), (255, 17), (40, 40)):
        psi[j] = phi[i]
    p = torch.from_numpy(phi).cuda().requires_grad_(True)
    q = torch.from_numpy(psi).cuda().requires_grad_(True)
    total, _ = functional.infonce_loss(p, q, "l2", loss, "mean", "row", 1.0, 0.1, "fused")
    total.backward()
    F = oracle.critic.energy_matrix(phi, psi, "l2", 1.0)
    G = oracle.critic.infonce_grad_F(F, loss, "mean", float(np.float32(0.1)), "row")
    want = oracle.critic.energy_backward(phi, psi, G, "l2", 1.0)
    # the coefficients are rounded to BF16 (relative 2^-9) before the products
    for got, ref in zip((p.grad, q.grad), want):
        got = got.double().cpu().numpy()
        assert np.isfinite(got).all()
        assert np.linalg.norm(got - ref) <= 2 ** -8 * np.linalg.norm(ref)
