"""The grouped GEMM's epilogues where their steps end inside a tile: hidden widths
that are no multiple of the 64- and 32-column steps, row blocks that end inside a
warp's 32 rows, and unaligned gradient rows (odd input widths).  The wide tiles
store through output tensor maps, the narrow ones by themselves: both must write
the same bits, and nothing outside their arrays."""

import numpy as np
import pytest
import torch

from paper_2408_11052_gb300 import api, workload

from parity_helpers import setup, small

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,B,layernorm", [(264, 136, False), (264, 136, True), (328, 40, False), (520, 392, False),
                                               (520, 264, True), (72, 8, False)])
def test_wide_and_narrow_tiles_store_the_same_bits(hidden, B, layernorm):
    """Two update steps on the one-tile (64-wide) and CTA-pair (256-wide where every width allows, else 128) kernels."""
    w = small(B=B, hidden=hidden, repr=64, E=8, T=300, layernorm=layernorm)
    prev_tune = api.set_autotune(False)
    runs = []
    try:
        for mode in ("one_tile", "cta_pair", "persistent"):
            prev = api.set_gemm_kernel(mode)
            try:
                ctx, _, _ = setup(w, precision="bf16", path="fused", n=200, mean_len=30.0)
                extra = workload.buffer_contents(w, n=2, mean_len=9.0, seed_offset=5)
                loss = torch.zeros(6, dtype=torch.float32, device=ctx.device)
                for i in range(2):
                    ctx.update_step(*(torch.from_numpy(x[i:i + 1]).to(ctx.device) for x in extra), loss_out=loss)
                torch.cuda.synchronize()
                assert ctx.sync_status() == (0, 0)
                runs.append([loss.cpu().numpy()] + [ctx.store[n][k].cpu().numpy() for n in ("phi", "psi", "pi")
                                                    for k in ("params", "grads")])
            finally:
                api.set_gemm_kernel(prev)
    finally:
        api.set_autotune(prev_tune)
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            np.testing.assert_array_equal(a, b)
