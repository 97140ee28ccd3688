"""A served request's admission footprint bounds the device memory that the
request holds at any time while it runs."""

import ctypes

import numpy as np
import pytest

import synth
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu

_USED, _USED_HIGH = 7, 8  # cudaMemPoolAttrUsedMemCurrent, cudaMemPoolAttrUsedMemHigh


class _Pool:
    """Counters of the device's default memory pool."""

    def __init__(self):
        self.rt = ctypes.CDLL("libcudart.so.13")
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def get(self, attr):
        v = ctypes.c_uint64()
        assert self.rt.cudaMemPoolGetAttribute(self.pool, attr, ctypes.byref(v)) == 0
        return v.value

    def restart(self):
        v = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolSetAttribute(self.pool, _USED_HIGH, ctypes.byref(v)) == 0
        return self.get(_USED)


def _ferromagnet(n):
    """All restarts end in one of two states of the same energy, so the final
    energy call takes its most candidates."""
    J = np.full((n, n), np.float32(0.1) / n)
    np.fill_diagonal(J, 0.0)
    return synth.Instance(n=n, layout="dense", J=J.astype(np.float32), name="ferromagnet")


def _case(name):
    if name == "many_restarts":  # the state outweighs the couplings; rows of whole lines
        return synth.sk_dense(2001, 1, 0.02, np.float32), dict(restarts=30000, steps=3, precision="tc")
    if name == "fp8_rows":
        return synth.er_dense(1930, 1, mean_degree=8, weights="pm1"), dict(restarts=30000, steps=3)
    if name == "sparse_slices":
        return (synth.random_sparse_instance(2000, 2, p=0.15, kind="float", h="zero"),
                dict(restarts=200, steps=20))
    if name == "sparse_int8":
        return (synth.random_sparse_instance(2000, 2, p=0.2, kind="int", h="zero", jmax=1),
                dict(restarts=200, steps=20))
    return _ferromagnet(2500), dict(restarts=64, steps=60, lr=1.0, precision="tc")


@pytest.mark.parametrize("name", ["many_restarts", "fp8_rows", "sparse_slices", "sparse_int8",
                                  "final_candidates"])
def test_footprint_bounds_the_memory_held(gpu_ctx, name):
    inst, kw = _case(name)
    gpu_ctx.synchronize()
    pool = _Pool()
    srv = api.Server(gpu_ctx, budget_bytes=64 << 30, max_active=1, chunk_steps=50, pack=False)
    before = pool.restart()
    res = srv.wait(srv.submit(inst, zero_rule=False, seed=1, **kw), timeout=300)
    assert res["status"] == 0, res["error"]
    held = pool.get(_USED_HIGH) - before
    srv.close()
    assert held <= res["footprint"], (held, res["footprint"])


def test_a_request_near_the_budget_is_still_accepted(gpu_ctx):
    """Its instance, operands and state fit; what pruning and the final energies
    may need beside them takes the rest of the budget, and it runs alone."""
    inst = synth.er_dense(2000, 1, mean_degree=8, weights="pm1")
    srv = api.Server(gpu_ctx, budget_bytes=40 << 20, max_active=2, chunk_steps=10)
    ids = [srv.submit(inst, restarts=128, steps=20, seed=k) for k in range(2)]
    a, b = [srv.wait(i, timeout=300) for i in ids]
    srv.close()
    assert a["status"] == 0 and b["status"] == 0
    assert a["footprint"] == b["footprint"] == 40 << 20
    assert b["t_admit_ms"] >= a["t_done_ms"] - 1e-6
