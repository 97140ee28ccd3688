"""Where a form's scratch finds no room, the call gives way to the form that
needs less, with the same results (the limit makes larger allocations fail)."""

import contextlib
import dataclasses

import numpy as np
import pytest
import torch

import synth
from oracle import ising
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def _limit(ctx, n):
    ctx.check(ctx.lib.ising_selftest_alloc_limit(ctx.handle, n))
    try:
        yield
    finally:
        ctx.check(ctx.lib.ising_selftest_alloc_limit(ctx.handle, 0))


def _device(inst):
    t = lambda x: None if x is None else torch.as_tensor(x).cuda()
    return dataclasses.replace(inst, J=t(inst.J), indptr=t(inst.indptr), indices=t(inst.indices),
                               data=t(inst.data), h=t(inst.h))


def test_limit_is_an_error_where_nothing_fits(gpu_ctx):
    inst = synth.sk_dense(200, 1, 1.0, np.float32)
    with _limit(gpu_ctx, 1000):
        with pytest.raises(api.IsingError) as e:
            api.energy(gpu_ctx, inst, np.ones((1, 200), np.int8))
    assert e.value.code == 2  # ISING_ENOMEM


@pytest.mark.parametrize("kind", ["int", "float"])
def test_packed_energies(gpu_ctx, kind):
    """A lane per vector needs the spins as bits (12 bytes per site for 65
    vectors), the general form partial sums (8.1 bytes per site each)."""
    n, count = 4096, 65
    a = np.arange(0, n, 2)
    e = np.stack([a, a + 1], 1)
    w = (1 + a % 5).astype(np.int8) if kind == "int" else np.sin(1.0 + a).astype(np.float32)
    ip, ix, da = synth.instances.csr_from_edges(n, e, w)
    inst = synth.Instance(n=n, layout="csr", indptr=ip, indices=ix, data=da.astype(w.dtype), name="pairs")
    s = (2 * np.random.default_rng(1).integers(0, 2, (count, n)) - 1).astype(np.int8)
    ref = np.asarray(ising.energy(inst, s.T), np.float64)
    with _limit(gpu_ctx, 10 * n):
        E = api.energy(gpu_ctx, _device(inst), torch.as_tensor(s).cuda())
    np.testing.assert_allclose(E.cpu().numpy(), ref, rtol=1e-12, atol=1e-10)


def test_digit_planes(gpu_ctx):
    n, count = 1100, 230
    inst = synth.sk_dense(n, 3, 1.0, np.float32)
    s = (2 * np.random.default_rng(2).integers(0, 2, (count, n)) - 1).astype(np.int8)
    ref = np.asarray(ising.energy(inst, s.T), np.float64)
    with _limit(gpu_ctx, 6 * n * n):  # the instance, and not its planes
        E = api.energy(gpu_ctx, _device(inst), torch.as_tensor(s).cuda())
    np.testing.assert_allclose(E.cpu().numpy(), ref, rtol=1e-12, atol=1e-9)


def test_sparse_session_without_room_for_its_slices(gpu_ctx):
    """FP32 couplings: 4 bytes each in every list but the slices (8 and padding)."""
    inst = synth.random_sparse_instance(900, 4, p=0.12, kind="float", h="zero")
    inst.data = inst.data.astype(np.float32)
    nnz = len(inst.data)
    kw = dict(restarts=3, steps=12, seed=5)
    with _limit(gpu_ctx, 6 * nnz):
        s = api.Session(gpu_ctx, inst, **kw)
        s.run(12)
        a, fa = s.restart_best(), s.result()["resident"]
        s.close()
    s = api.Session(gpu_ctx, inst, **kw)
    s.run(12)
    b, fb = s.restart_best(), s.result()["resident"]
    s.close()
    assert (fa, fb) == (0, 3)
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)
