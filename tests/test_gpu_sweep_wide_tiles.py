"""Grouped sweeps at repr 192 and 256, whose output layers run on 256-wide tiles: one
warp of the kernels that walk the problem list takes a policy's output (which leaves
its staging block as TMA stores where the rows allow it, A a multiple of 2), then an
encoder's or another policy's, which it stores itself out of the same block.  More
tiles than SMs, so that every CTA takes several; bit for bit the agents alone, whose
lists never put the one kind after the other."""

import pytest

from paper_2408_11052_gb300 import api, workload

from test_gpu_sweep import run_and_compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["persistent", "cta_pair", "one_tile"])
@pytest.mark.parametrize("repr_", [192, 256])
def test_policy_and_encoder_outputs_share_wide_tiles(mode, repr_):
    acts = (8, 17, 16, 8, 17, 8, 16, 17, 8)
    ws = [workload.Workload(f"wide{i}", E=12, T=60, D=29, A=A, G=2, B=2048 - 136 * (i % 3), hidden=64, layers=2,
                            repr=repr_, seed=60 + i) for i, A in enumerate(acts)]
    prev_tune, prev = api.set_autotune(False), api.set_gemm_kernel(mode)
    try:
        run_and_compare(ws, "bf16", "fused", grouped=True, steps=6)
    finally:
        api.set_gemm_kernel(prev)
        api.set_autotune(prev_tune)
