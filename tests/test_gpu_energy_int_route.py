"""Energies of dense integer instances on both sides of the rule that chooses
between the general and the fixed form by size and vectors: exact in each."""

import numpy as np
import pytest

import synth
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.int8, np.float64])
@pytest.mark.parametrize("n,counts", [(3, (1, 700)), (150, (1, 16, 300)), (160, (1, 15, 300)),
                                      (255, (1, 100, 140, 900)), (384, (16, 250, 330)),
                                      (636, (2, 400)), (637, (1, 64)), (1000, (1, 5, 20))])
def test_integers_are_exact(gpu_ctx, dtype, n, counts):
    inst = synth.random_sparse_instance(n, n, p=0.7, kind="int", h="int", layout="dense", jmax=100)
    inst.J = inst.J.astype(dtype)
    J = np.asarray(inst.J, np.float64)
    for count in counts:
        s = (2 * np.random.default_rng(count).integers(0, 2, (count, n)) - 1).astype(np.int8)
        E, Q, H = api.energy(gpu_ctx, inst, s, exact_parts=True)
        x = s.astype(np.float64)  # (sums below 2^53: exact in any order)
        np.testing.assert_array_equal(Q, ((x @ J) * x).sum(1).astype(np.int64))
        np.testing.assert_array_equal(H, (x @ np.asarray(inst.h, np.float64)).astype(np.int64))
