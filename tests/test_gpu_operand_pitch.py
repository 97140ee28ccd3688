"""Tensor-core operands whose rows are padded to whole 128-byte lines (where
that adds at most 1/16) and their neighbours that are not: coupling products
of integer couplings are exact, and a state survives export and import."""

import numpy as np
import pytest

import synth
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu


# 16-bit rows: 416 and 449 keep their pitch (6.5 and 7 lines), 417 to 440 take 448;
# 8-bit rows: 480 keeps 480, 481 to 496 take 512
@pytest.mark.parametrize("n,top", [(416, 100), (417, 100), (430, 100), (440, 100), (449, 100),
                                   (480, 1), (481, 1), (490, 1), (496, 1), (497, 1)])
@pytest.mark.parametrize("streaming", [False, True])
def test_products_and_state_at_each_pitch(gpu_ctx, n, top, streaming):
    rng = np.random.default_rng(n)
    inst = synth.er_dense(n, n, p=0.3, weights="pm1")
    J = np.triu(rng.integers(-top, top + 1, (n, n)), 1)
    inst.J = (J + J.T).astype(np.asarray(inst.J).dtype)
    s = api.Session(gpu_ctx, inst, restarts=70, steps=8, seed=3, streaming=streaming)
    s.run(3)
    st = s.export_state()
    sp = st["spins"].astype(np.int64)
    np.testing.assert_array_equal(s.coupling(), (sp @ inst.J.astype(np.int64)).astype(np.float32))
    o = api.Session(gpu_ctx, inst, restarts=70, steps=8, seed=9, streaming=streaming)
    o.import_state(st["theta"], st["m"], st["v"], st["t"])
    s.run(5)
    o.run(5)
    a, b = s.export_state(), o.export_state()
    for k in ["theta", "m", "v", "spins"]:
        np.testing.assert_array_equal(a[k], b[k])
    s.close()
    o.close()
