"""GPU parity of the linear-message kernels and of what stands behind them: gradients of any scale, outputs in place, blocks
without a certificate, which kernels a call runs."""
import numpy as np
import pytest

import oracle
import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2605_10655_b200 import Context
    c = Context(0)
    yield c
    c.close()


def _rand(n, Lb, B, seed):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal((B, n)).astype(np.float32), rng.standard_normal(1 << Lb).astype(np.float32),
            rng.standard_normal((B, n)).astype(np.float32))


@pytest.mark.parametrize("messages", [0, 1], ids=["linear", "log"])
@pytest.mark.parametrize("Lb,B", [(8, 4000), (9, 2500)])
def test_one_warp_blocks_start_from_their_own_first_step(ctx, Lb, B, messages):
    # One warp per block, more blocks than fit at once: the alpha sweep's initial messages hold the first step's gradient term, which
    # lane 0 has just written.  Only the first weight has an upstream gradient, and it alternates in sign and size from block to block.
    n, T = 3, 0.3
    W, c, g = _rand(n, Lb, B, seed=600 + Lb)
    g[:] = 0.0
    g[:, 0] = np.where(np.arange(B) % 2 == 0, 1.0, -1.0) * (1.0 + np.arange(B) % 7)
    ctx.set_option("messages", messages)
    try:
        got = parity.gpu_forward_backward(ctx, W, c, g, Lb, 2, T)
    finally:
        ctx.set_option("messages", 0)
    assert got["diag"].device_status == 0
    ref_b = oracle.backward(W, c, g, Lb, 2, T)
    assert parity.rel_inf(got["grad_W"], ref_b["grad_W"]) <= 1e-5          # three float32 steps
    assert parity.rel_inf(got["grad_codebook"], ref_b["grad_codebook"]) <= 1e-5
