"""ising_ds_stats.resident names the form that a sparse session took, and each
variant of the resident form (spins as words or bits, couplings on chip or
not, by value type) equals a launch per step bit for bit."""

import numpy as np
import pytest

import synth
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu


def _ring(n, kind, extra=0):
    """A ring with `extra` further neighbours per spin."""
    a = np.repeat(np.arange(n), 1 + extra)
    b = (a + np.tile(1 + 7 * np.arange(1 + extra), n)) % n
    e = np.unique(np.stack([np.minimum(a, b), np.maximum(a, b)], 1), axis=0)
    k = np.arange(len(e))
    w = (np.where(k % 3, 1, -1) * (1 + k % 4)).astype(np.int32) if kind == "int" else np.sin(1.0 + k)
    ip, ix, da = synth.instances.csr_from_edges(n, e, w)
    return synth.Instance(n=n, layout="csr", indptr=ip, indices=ix, data=da, name="ring")


def _run(ctx, inst, B, T, **kw):
    s = api.Session(ctx, inst, restarts=B, steps=T, seed=3, **kw)
    s.run(T - 1)
    st = s.export_state()
    s.finish()
    best, last, res = s.restart_best(), s.last_energies(), s.result()
    s.close()
    return st, best, last, res


# spins as words fit up to about 14300 / restarts per CTA, as bits up to 16300;
# couplings stay in device memory where the state leaves no room for them
_BOTH = [(200, 1, 3), (9000, 6, 3), (14500, 1, 2), (14800, 3, 1), (7200, 2, 200), (7800, 6, 160)]
_INT = [(16300, 3, 1), (3300, 12, 500), (3640, 2, 400), (1800, 4, 1300), (2000, 140, 152)]


@pytest.mark.parametrize("kind,n,extra,B", [(k, *c) for c in _BOTH for k in ("int", "float")] +
                         [("int", *c) for c in _INT])
def test_resident_variants(gpu_ctx, kind, n, extra, B):
    inst = _ring(n, kind, extra)
    a = _run(gpu_ctx, inst, B, 14)
    b = _run(gpu_ctx, inst, B, 14, streaming=True, autotune=False)
    assert (a[3]["resident"], b[3]["resident"]) == (3, 0)
    for k in ("theta", "m", "v", "spins"):
        np.testing.assert_array_equal(a[0][k], b[0][k])
    for x, y in zip(a[1], b[1]):
        np.testing.assert_array_equal(x, y)
    np.testing.assert_array_equal(a[2], b[2])
    assert a[3]["best_energy"] == b[3]["best_energy"]


# instances that the form declines: too many spins for shared memory, more
# sites and restarts per thread than a word has bits, couplings that few restarts'
# CTAs would walk too long, threads with many rows each, a row that would pad its
# slice far beyond the others, the relaxed product
@pytest.mark.parametrize("case", ["large", "large_float", "bits", "few", "few_float", "rows", "hub",
                                  "relaxed"])
def test_declined(gpu_ctx, case):
    kw, B = {}, 4
    if case == "large":
        inst, B = _ring(16500, "int", 3), 1
    elif case == "large_float":
        inst, B = _ring(16500, "float", 3), 1
    elif case == "bits":
        inst, B = _ring(3300, "float", 12), 500
    elif case == "few":
        inst, B = _ring(2000, "int", 140), 8
    elif case == "few_float":
        inst, B = _ring(9000, "float", 12), 8
    elif case == "rows":
        inst, B, kw = _ring(300, "float", 23), 16384, dict(converge=True)
    elif case == "hub":
        n = 6000
        e = np.stack([np.zeros(n - 1, np.int64), np.arange(1, n)], 1)
        ip, ix, da = synth.instances.csr_from_edges(n, e, np.ones(len(e), np.int32))
        inst = synth.Instance(n=n, layout="csr", indptr=ip, indices=ix, data=da, name="star")
    else:
        inst, kw = _ring(300, "float"), dict(relaxed=True)
    s = api.Session(gpu_ctx, inst, restarts=B, steps=3, seed=3, **kw)
    s.run(3)
    assert s.result()["resident"] == 0
    s.close()
