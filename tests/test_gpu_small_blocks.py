"""The small tensor-core form (n <= 128) at the edges of its blocks of 16, 32,
64 and 128 restarts (the narrowest that one wave of 152 SMs holds): state,
bests and energies are those of the streaming form bit for bit."""

import numpy as np
import pytest

import synth
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,prec", [("pm1", 128, "fp8"), ("pm1", 3, "auto"), ("float", 65, "tc")])
@pytest.mark.parametrize("B", [1, 15, 16, 17, 2432, 2433, 4865, 9729])
def test_small_blocks_equal_streaming(gpu_ctx, kind, n, prec, B):
    inst = (synth.er_dense(n, 31, p=0.5, weights="pm1") if kind == "pm1"
            else synth.sk_dense(n, 32, 0.2, np.float32, h_std=0.4))
    a = api.Session(gpu_ctx, inst, restarts=B, steps=9, seed=5, precision=prec)
    b = api.Session(gpu_ctx, inst, restarts=B, steps=9, seed=5, precision=prec, streaming=True)
    a.run(4)
    a.run(5)
    b.run(9)
    sa, sb = a.export_state(), b.export_state()
    for k in ["theta", "m", "v", "spins"]:
        np.testing.assert_array_equal(sa[k], sb[k])
    for x, y in zip(a.restart_best(), b.restart_best()):
        np.testing.assert_array_equal(x, y)
    np.testing.assert_array_equal(a.last_energies(), b.last_energies())
    a.close()
    b.close()
