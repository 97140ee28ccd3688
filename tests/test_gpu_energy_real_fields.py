"""Dense integer couplings beside fields that are not dyadic: the couplings'
part of the energy is an exact integer, the fields' an FP64 sum."""

import numpy as np
import pytest

import synth
from oracle import ising
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _reference(inst, s):
    cq, ch = ising.coefficients(inst.j_scale, inst.convention)
    J, x = np.asarray(inst.J, np.int64), s.astype(np.int64)
    Q = ((x @ J) * x).sum(1)
    ref = np.longdouble(cq) * Q + np.longdouble(ch) * (s.astype(np.longdouble) @ np.asarray(inst.h, np.longdouble))
    # Q is exact; its product, the sum of n field terms and the last addition round
    bound = EPS * (4 * abs(cq) * np.abs(Q) + (inst.n + 4) * abs(ch) * np.abs(inst.h).sum())
    return ref, bound


# one vector and several (fixed form), many (digit planes from 2^28 coupling-vectors on)
@pytest.mark.parametrize("dtype", [np.int8, np.int32, np.float32, np.float64])
@pytest.mark.parametrize("n,count", [(5, 1), (131, 3), (132, 4), (1030, 1), (1030, 260)])
def test_integer_couplings_with_real_fields(gpu_ctx, dtype, n, count):
    inst = synth.random_sparse_instance(n, 2, p=0.4, kind="int", h="float", layout="dense",
                                        jmax=100 if dtype == np.int8 else 100000)
    inst.J = inst.J.astype(dtype)
    r = np.random.default_rng(n + count)
    s = (2 * r.integers(0, 2, (count, n)) - 1).astype(np.int8)
    ref, bound = _reference(inst, s)
    assert np.all(np.abs(api.energy(gpu_ctx, inst, s) - ref) <= bound)


def test_smallest_int32_coupling(gpu_ctx):
    """|J| = 2^31 leaves the exact integer form, but stays an integer."""
    inst = synth.random_sparse_instance(40, 2, p=0.4, kind="int", h="float", layout="dense", jmax=100)
    inst.J = inst.J.astype(np.int32)
    inst.J[3, 9] = inst.J[9, 3] = -2 ** 31
    s = (2 * np.random.default_rng(1).integers(0, 2, (6, 40)) - 1).astype(np.int8)
    ref, bound = _reference(inst, s)
    assert np.all(np.abs(api.energy(gpu_ctx, inst, s) - ref) <= bound)


def test_solve_reports_the_energy_of_its_spins(gpu_ctx):
    inst = synth.random_sparse_instance(100, 3, p=0.5, kind="int", h="float", layout="dense", jmax=3)
    inst.J = inst.J.astype(np.int8)
    res = api.solve(gpu_ctx, inst, restarts=64, steps=60, seed=2)
    ref, bound = _reference(inst, res["best_spins"][None].astype(np.int8))
    assert abs(res["best_energy"] - ref[0]) <= bound[0]
