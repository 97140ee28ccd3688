"""Energies of many vectors on CSR instances with long rows, bounded by the
depth of the sums that a warp per row and vector forms."""

import numpy as np
import pytest

import synth
from oracle import ising
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _csr(n, edges, w):
    ip, ix, da = synth.instances.csr_from_edges(n, np.asarray(edges), np.asarray(w))
    return synth.Instance(n=n, layout="csr", indptr=ip, indices=ix, data=da, name="rows")


def _graph(kind, n):
    i, j = np.triu_indices(n, 1)
    if kind == "complete":
        e = np.stack([i, j], 1)
    elif kind == "star":
        e = np.stack([np.zeros(n - 1, np.int64), np.arange(1, n)], 1)
    else:  # circulant: rows of exactly `kind` entries
        k = int(kind) // 2
        a = np.repeat(np.arange(n), k)
        b = (a + np.tile(np.arange(1, k + 1), n)) % n
        e = np.unique(np.stack([np.minimum(a, b), np.maximum(a, b)], 1), axis=0)
    return e


def _check(ctx, inst, s):
    """A lane adds every 32nd entry of a row, five levels join the lanes, a
    warp adds eight rows and a block eight warps, then the blocks' partials
    are added 32 at a time and joined: no term passes through more roundings."""
    cq, _ = ising.coefficients(inst.j_scale, inst.convention)
    rows = np.repeat(np.arange(inst.n), np.diff(inst.indptr))
    J = np.asarray(inst.data, np.longdouble)
    x = s.astype(np.longdouble)
    ref = np.array([cq * (J * v[rows] * v[inst.indices]).sum() for v in x])
    longest = int(np.diff(inst.indptr).max())
    depth = -(-longest // 32) + 5 + 8 + 8 + -(-(-(-inst.n // 64)) // 32) + 5 + 2
    bound = EPS * depth * abs(cq) * float(np.abs(J).sum())
    assert np.all(np.abs(api.energy(ctx, inst, s) - ref) <= bound)


# equal couplings and spins: every rounding of a sum has the same sign
@pytest.mark.parametrize("value", [0.1, 1.0 / 3.0, 1.1])
@pytest.mark.parametrize("kind,n", [("complete", 600), ("complete", 1200), ("star", 20000),
                                    ("32", 500), ("34", 500), ("64", 500)])
@pytest.mark.parametrize("count", [8, 33])
def test_equal_terms(gpu_ctx, value, kind, n, count):
    e = _graph(kind, n)
    s = np.ones((count, n), np.int8)
    s[1::2, : n // 3] = -1
    _check(gpu_ctx, _csr(n, e, np.full(len(e), value)), s)


# many vectors of short and middling rows, a lane per vector: around the limits of
# the longest row (128, and twice the vectors) and of the work
@pytest.mark.parametrize("degree,count", [(2, 32), (30, 33), (32, 70), (64, 33), (66, 33), (68, 33),
                                          (128, 64), (130, 70)])
def test_equal_terms_a_lane_per_vector(gpu_ctx, degree, count):
    n = 2050
    e = _graph(str(degree), n)
    s = np.ones((count, n), np.int8)
    s[1::2, : n // 3] = -1
    _check(gpu_ctx, _csr(n, e, np.full(len(e), 1.0 / 3.0)), s)


@pytest.mark.parametrize("degree,count", [(2, 66), (64, 64), (66, 66), (70, 66), (128, 130), (130, 130)])
def test_integers_around_the_row_limit(gpu_ctx, degree, count):
    n = 4100
    e = _graph(str(degree), n)
    w = (1 + np.arange(len(e)) % 5).astype(np.int32)
    inst = _csr(n, e, w)
    r = np.random.default_rng(degree)
    s = (2 * r.integers(0, 2, (count, n)) - 1).astype(np.int8)
    E, Q, _ = api.energy(gpu_ctx, inst, s, exact_parts=True)
    Eo, Qo, _ = ising.energy_exact(inst, s.T)
    np.testing.assert_array_equal(Q, Qo)
    np.testing.assert_array_equal(E, Eo)


@pytest.mark.parametrize("kind", ["int", "float"])
@pytest.mark.parametrize("n,mean,count", [(9000, 1.5, 33), (9000, 6, 40), (4100, 21, 65)])
def test_rows_of_all_lengths(gpu_ctx, kind, n, mean, count):
    inst = synth.random_sparse_instance(n, 5, p=mean / n, kind=kind, h=kind)
    r = np.random.default_rng(n)
    s = (2 * r.integers(0, 2, (count, n)) - 1).astype(np.int8)
    if kind == "int":
        E, Q, H = api.energy(gpu_ctx, inst, s, exact_parts=True)
        Eo, Qo, Ho = ising.energy_exact(inst, s.T)
        np.testing.assert_array_equal(Q, Qo)
        np.testing.assert_array_equal(H, Ho)
        np.testing.assert_array_equal(E, Eo)
        return
    cq, ch = ising.coefficients(inst.j_scale, inst.convention)
    rows = np.repeat(np.arange(n), np.diff(inst.indptr))
    J, h, x = (np.asarray(v, np.longdouble) for v in (inst.data, inst.h, s))
    ref = np.array([cq * (J * v[rows] * v[inst.indices]).sum() + ch * (h * v).sum() for v in x])
    depth = 6 + 8 + 8 + -(-(-(-n // 64)) // 32) + 5 + 3
    bound = EPS * depth * (abs(cq) * float(np.abs(J).sum()) + abs(ch) * float(np.abs(h).sum()))
    assert np.all(np.abs(api.energy(gpu_ctx, inst, s) - ref) <= bound)
