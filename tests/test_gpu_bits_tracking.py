"""Best tracking of bit-packed spins beyond 4096 per restart (launch-per-step
sparse form): an improved restart's spins are copied by the next step's
tracking launch, the last step's at the end of a run. Every restart's best
spins have its best energy, whatever the run is cut into."""

import numpy as np
import pytest

import synth
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,B,converge", [(69, 1, False), (69, 33, False), (64, 300, False),
                                             (69, 300, True)])
def test_best_spins_have_the_best_energy(gpu_ctx, rows, B, converge):
    inst = synth.torus_csr(rows, 65, 5)  # 4160 or 4485 spins, integer couplings
    T = 110
    kw = dict(restarts=B, steps=T, seed=7, streaming=True, converge=converge)
    a = api.Session(gpu_ctx, inst, **kw)
    b = api.Session(gpu_ctx, inst, **kw)
    for k in (1, 2, 3):
        a.run(k)
        e, _, s = a.restart_best()[:3]
        np.testing.assert_array_equal(api.energy(gpu_ctx, inst, s), e)
    a.run(T - 6)
    b.run(T)
    for x, y in zip(a.restart_best(), b.restart_best()):
        np.testing.assert_array_equal(x, y)
    a.finish()
    e, _, s = a.restart_best()[:3]
    np.testing.assert_array_equal(api.energy(gpu_ctx, inst, s), e)
    a.close()
    b.close()
