"""The plain FP32 form at the edges of its tiles (128 spins x 32 to 128
restarts, 16 k per chunk, rows on and off 16-byte boundaries): its coupling
product is the FP32 sum in order of k, whatever the tile width."""

import numpy as np
import pytest

import synth
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu


def _in_order(J, s):
    """G[b][i]: FP32 accumulation over k in order of the products J_ik s_bk
    (+-J_ik exactly, so each step is one rounded addition)."""
    G = np.zeros((s.shape[0], J.shape[0]), np.float32)
    for k in range(J.shape[1]):
        G = (G + (s[:, k, None] * J[None, :, k]).astype(np.float32)).astype(np.float32)
    return G


# restart counts that make each width the least waves of tiles on 152 SMs for
# one to three row tiles, with ragged last tiles
@pytest.mark.parametrize("n", [1, 15, 16, 17, 100, 129, 300])
@pytest.mark.parametrize("B", [1, 31, 50, 4864, 9000])
def test_product_is_the_ordered_sum(gpu_ctx, n, B):
    if n * B > 1000000:
        B = 4864
    inst = synth.sk_dense(n, 3 + n, 1.0, np.float32, h_std=0.5)
    s = api.Session(gpu_ctx, inst, restarts=B, steps=3, seed=2, precision="fp32")
    s.run(1)
    sp = s.export_state()["spins"].astype(np.float32)
    np.testing.assert_array_equal(s.coupling(), _in_order(inst.J.astype(np.float32), sp))
    s.close()
