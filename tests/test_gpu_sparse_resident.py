"""Sparse resident form (all steps of a run in one launch, a few restarts per
CTA) against the launch-per-step form (streaming=True), bit for bit: state,
spins, bests, energies and the convergence rule, at the edges of its layout."""

import numpy as np
import pytest

import synth
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu


def _hub(n):
    """A star on top of a ring: one row longer than all others."""
    e = [(0, j) for j in range(2, n - 1)] + [(j, j + 1) for j in range(n - 1)] + [(0, n - 1)]
    e = np.unique(np.array(e), axis=0)
    w = (1 + np.arange(len(e)) % 3).astype(np.int32) * np.where(np.arange(len(e)) % 2, 1, -1).astype(np.int32)
    ip, ix, da = synth.instances.csr_from_edges(n, e, w)
    return synth.Instance(n=n, layout="csr", indptr=ip, indices=ix, data=da, name="hub")


INSTANCES = {
    "one": synth.random_sparse_instance(1, 1, kind="int", h="int"),
    "no_edges": synth.random_sparse_instance(40, 1, p=0.0, kind="float", h="float"),
    "torus": synth.torus_csr(10, 13, 5),
    "int_h": synth.random_sparse_instance(333, 2, p=0.02, kind="int", h="int", convention="paper"),
    "int_large": synth.random_sparse_instance(150, 3, p=0.1, kind="int", h="zero", jmax=1000),
    "int8_float_h": synth.random_sparse_instance(150, 3, p=0.1, kind="int", h="float"),
    "float": synth.random_sparse_instance(257, 7, p=0.05, kind="float", h="float"),
    "float_two_passes": synth.random_sparse_instance(1800, 8, p=0.004, kind="float", h="zero"),
    "er": synth.random_sparse_instance(2100, 9, p=0.004, kind="int", h="zero", jmax=1),
    "hub": _hub(70),
}


def _pair(ctx, inst, B, T, **kw):
    return (api.Session(ctx, inst, restarts=B, steps=T, seed=7, **kw),
            api.Session(ctx, inst, restarts=B, steps=T, seed=7, streaming=True, autotune=False, **kw))


def _same(a, b, state=True):
    if state:
        sa, sb = a.export_state(), b.export_state()
        for k in ("theta", "m", "v", "spins"):
            np.testing.assert_array_equal(sa[k], sb[k])
        assert sa["t"] == sb["t"]
    np.testing.assert_array_equal(a.last_energies(), b.last_energies())
    for x, y in zip(a.restart_best(), b.restart_best()):
        np.testing.assert_array_equal(x, y)


# restarts per CTA: 1, 2, 4 and 8 (one wave and several), the last block ragged
@pytest.mark.parametrize("name", INSTANCES)
@pytest.mark.parametrize("B", [1, 33, 153, 305, 700, 1300])
def test_equals_launch_per_step(gpu_ctx, name, B):
    inst = INSTANCES[name]
    if inst.n > 1000 and B > 400:
        B = 305
    a, b = _pair(gpu_ctx, inst, B, 40, mu=0.1)
    for k in (1, 2, 24):  # runs of one, two and more steps
        a.run(k)
        b.run(k)
        _same(a, b)
    np.testing.assert_array_equal(a.coupling(), b.coupling())
    a.finish()
    b.finish()
    _same(a, b, state=False)
    ra, rb = a.result(), b.result()
    for k in ("best_energy", "best_restart", "best_step", "last_best_energy"):
        assert ra[k] == rb[k]
    assert a.work() == b.work()
    a.close()
    b.close()


@pytest.mark.parametrize("name", ["torus", "float", "int_h"])
@pytest.mark.parametrize("B,lr", [(40, 0.05), (520, 6.0), (520, 0.0)])
def test_convergence_rule(gpu_ctx, name, B, lr):
    a, b = _pair(gpu_ctx, INSTANCES[name], B, 260, lr=lr, converge=True)
    for s in (a, b):
        s.run(7)
        s.run(260)
        s.finish()
    np.testing.assert_array_equal(a.convergence(), b.convergence())
    _same(a, b, state=False)
    assert a.work() == b.work()
    a.close()
    b.close()


def test_imported_state(gpu_ctx):
    inst = INSTANCES["float"]
    rng = np.random.default_rng(1)
    th, m = rng.uniform(-3, 3, (50, inst.n)), rng.normal(size=(50, inst.n))
    v = rng.uniform(0.01, 1, (50, inst.n))
    a, b = _pair(gpu_ctx, inst, 50, 30)
    for s in (a, b):
        s.run(3)
        s.import_state(th, m, v, 11)
        s.run(9)
    _same(a, b)
    a.close()
    b.close()
