"""The forms of the energy kernel at the edges of their tiles: dense couplings
as fixed-point integers (rows in fours, columns in groups of 32 or 128, one or
several vectors per pass), CSR with 32 vectors per warp, and the cases left to
the general form."""

import numpy as np
import pytest

import synth
from oracle import ising
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _spins(count, n, seed):
    r = np.random.default_rng(seed)
    return (2 * r.integers(0, 2, (count, n)) - 1).astype(np.int8)


def _check_float(ctx, inst, s):
    """Against extended precision. The couplings' roundings add up to at most
    16 eps sum |J|, the rest is a handful of FP64 roundings of the two sums,
    the field's sum of n terms one per term."""
    cq, ch = ising.coefficients(inst.j_scale, inst.convention)
    J = np.asarray(inst.J, np.longdouble)
    h = np.zeros(inst.n, np.longdouble) if inst.h is None else np.asarray(inst.h, np.longdouble)
    x = s.astype(np.longdouble)
    ref = cq * ((x @ J) * x).sum(1) + ch * (x @ h)
    bound = EPS * ((16 + 8) * abs(cq) * np.abs(J).sum() + (inst.n + 8) * np.abs(h).sum())
    E = api.energy(ctx, inst, s)
    assert np.all(np.abs(E - ref) <= np.asarray(bound, np.float64) + 1e-300)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n", [1, 3, 4, 31, 128, 129, 1023, 1028])
@pytest.mark.parametrize("count", [1, 4, 5])
def test_dense_float(gpu_ctx, dtype, n, count):
    inst = synth.sk_dense(n, n, 1.0, dtype, h_std=0.3)
    _check_float(gpu_ctx, inst, _spins(count, n, n + count))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n,count", [(520, 1000), (1025, 300), (2050, 70), (4100, 17)])
def test_dense_many_vectors(gpu_ctx, dtype, n, count):
    """Digits in planes: 12 bits each up to n = 2048, 11 and 10 beyond (a
    sampled subset of the vectors is checked)."""
    inst = synth.sk_dense(n, n, 1.0, dtype, h_std=0.3)
    s = _spins(count, n, n + count)
    E = api.energy(gpu_ctx, inst, s)
    pick = np.unique(np.linspace(0, count - 1, 12).astype(int))
    cq, ch = ising.coefficients(inst.j_scale, inst.convention)
    J, h = np.asarray(inst.J, np.longdouble), np.asarray(inst.h, np.longdouble)
    x = s[pick].astype(np.longdouble)
    ref = cq * ((x @ J) * x).sum(1) + ch * (x @ h)
    bound = EPS * (24 * abs(cq) * np.abs(J).sum() + (n + 8) * np.abs(h).sum())
    assert np.all(np.abs(E[pick] - ref) <= float(bound))
    # one vector at a time takes the fixed form: the same integers up to the scale
    one = np.array([api.energy(gpu_ctx, inst, s[k:k + 1])[0] for k in pick[:3]])
    assert np.all(np.abs(one - E[pick[:3]]) <= float(bound))


@pytest.mark.parametrize("dtype", [np.int8, np.int32, np.float32])
def test_dense_integers_many_vectors(gpu_ctx, dtype):
    n, count = 1030, 260
    inst = synth.random_sparse_instance(n, 2, p=0.3, kind="int", h="int", layout="dense",
                                        jmax=100 if dtype == np.int8 else 100000)
    inst.J = inst.J.astype(dtype)
    s = _spins(count, n, 1)
    ref = synth.Instance(n=n, layout="dense", J=inst.J.astype(np.int32), h=inst.h,
                         j_scale=inst.j_scale, convention=inst.convention)
    E, Q, H = api.energy(gpu_ctx, inst, s, exact_parts=True)
    Eo, Qo, Ho = ising.energy_exact(ref, s.T)
    np.testing.assert_array_equal(Q, Qo)
    np.testing.assert_array_equal(H, Ho)
    np.testing.assert_array_equal(E, Eo)


@pytest.mark.parametrize("scale", [1e-30, 1.0, 3e28])
def test_dense_float_scales(gpu_ctx, scale):
    inst = synth.sk_dense(260, 5, 1.0, np.float32)
    inst.J = (inst.J * np.float32(scale)).astype(np.float32)
    _check_float(gpu_ctx, inst, _spins(3, 260, 9))


def test_dense_wide_range(gpu_ctx):
    """One coupling 2^90 above the others: no single scale holds them."""
    inst = synth.sk_dense(200, 6, 1.0, np.float64)
    inst.J[3, 7] = inst.J[7, 3] = 2.0 ** 90
    _check_float(gpu_ctx, inst, _spins(3, 200, 9))


@pytest.mark.parametrize("dtype", [np.int8, np.int32, np.float32, np.float64])
@pytest.mark.parametrize("n", [5, 132, 515])
def test_dense_integers_are_exact(gpu_ctx, dtype, n):
    inst = synth.random_sparse_instance(n, n, p=0.7, kind="int", h="int", layout="dense", jmax=100)
    inst.J = inst.J.astype(dtype)
    s = _spins(6, n, 1)
    ref = synth.Instance(n=n, layout="dense", J=inst.J.astype(np.int32), h=inst.h,
                         j_scale=inst.j_scale, convention=inst.convention)
    E, Q, H = api.energy(gpu_ctx, inst, s, exact_parts=True)
    Eo, Qo, Ho = ising.energy_exact(ref, s.T)
    np.testing.assert_array_equal(Q, Qo)
    np.testing.assert_array_equal(H, Ho)
    np.testing.assert_array_equal(E, Eo)


@pytest.mark.parametrize("count", [7, 8, 31, 33, 64])
@pytest.mark.parametrize("kind", ["int", "float"])
def test_csr_vectors(gpu_ctx, count, kind):
    n = 197
    inst = synth.random_sparse_instance(n, 3, p=0.05, kind=kind, h=kind)
    s = _spins(count, n, count)
    if kind == "int":
        E, Q, H = api.energy(gpu_ctx, inst, s, exact_parts=True)
        Eo, Qo, Ho = ising.energy_exact(inst, s.T)
        np.testing.assert_array_equal(Q, Qo)
        np.testing.assert_array_equal(H, Ho)
        np.testing.assert_array_equal(E, Eo)
    else:
        np.testing.assert_allclose(api.energy(gpu_ctx, inst, s), ising.energy(inst, s.T), rtol=1e-12,
                                   atol=1e-10)


@pytest.mark.parametrize("layout", ["dense", "csr"])
def test_spins_other_than_pm1(gpu_ctx, layout):
    """The quadratic form of any int8 vectors, as before the bit forms."""
    inst = synth.random_sparse_instance(90, 4, p=0.3, kind="int", h="int", layout=layout)
    s = _spins(9, 90, 2)
    s[2, 5], s[4, 80] = 0, 3
    J = np.asarray(inst.dense(), np.int64)
    x = s.astype(np.int64)
    _, Q, H = api.energy(gpu_ctx, inst, s, exact_parts=True)
    np.testing.assert_array_equal(Q, ((x @ J) * x).sum(1))
    np.testing.assert_array_equal(H, x @ inst.h.astype(np.int64))
