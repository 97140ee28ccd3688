"""Pair-MMA tiles of several widths (several waves per CTA pair, tiles cut at row
tiles, a last unit of 32 restarts that a wave gives away) against single-CTA
tiles of 128, and the grid-wide resident form with one group of 32 or 64 restarts
and with couplings that stream through its ring against a launch per step: bit
for bit."""

import math

import numpy as np
import pytest

import synth
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu


def _run(ctx, inst, B, T, shape=None, **kw):
    s = api.Session(ctx, inst, restarts=B, steps=T, seed=8, autotune=False, **kw)
    if shape is not None:
        s.set_tiles(*shape)
    s.run(T)
    st = s.export_state()
    best = s.restart_best()
    s.finish()
    last, res = s.last_energies(), s.result()
    s.close()
    return st, best, last, res


def _same(a, b):
    for k in ("theta", "m", "v", "spins"):
        np.testing.assert_array_equal(a[0][k], b[0][k], err_msg=k)
    for x, y in zip(a[1], b[1]):
        np.testing.assert_array_equal(x, y)
    np.testing.assert_array_equal(a[2], b[2])
    assert a[3]["best_energy"] == b[3]["best_energy"]


def _instance(kind, n):
    if kind == "e4m3":
        return synth.er_dense(n, 53, mean_degree=8, weights="pm1")
    return synth.sk_dense(n, 51, 1 / math.sqrt(n), np.float32, h_std=0.3)


# units of 32 restarts per pair (76 pairs): 1 pair row of 130 spins takes 8, 9, 15,
# 17 and 3; 3 pair rows of 520 spins 9 (cut at rows, ragged) and 18
@pytest.mark.parametrize("kind", ["two_planes", "e4m3"])
@pytest.mark.parametrize("n,B", [(130, 32 * 76 * 8), (130, 32 * 76 * 8 + 5), (130, 32 * 76 * 15 - 40),
                                 (130, 32 * 76 * 17), (130, 32 * 76 * 3 - 31), (520, 6517), (520, 14001)])
def test_widths_are_bit_identical(gpu_ctx, kind, n, B):
    inst = _instance(kind, n)
    ref = _run(gpu_ctx, inst, B, 5, (128, 0), streaming=True)
    for bn in (224, 256):
        got = _run(gpu_ctx, inst, B, 5, (bn, 2), streaming=True)
        assert (got[3]["tile_restarts"], got[3]["tile_pair"]) == (bn, 2)
        _same(got, ref)


# restarts per group: 32, 64 and two of 64 (152 SMs over the row tiles); 1000 spins
# in two planes and 1900, 2000 in one have more units than stay in shared memory
@pytest.mark.parametrize("kind,n,B", [
    ("two_planes", 1000, 600), ("two_planes", 1000, 1201), ("two_planes", 1000, 2400),
    ("two_planes", 300, 1500), ("e4m3", 1900, 300), ("e4m3", 1900, 600), ("e4m3", 2000, 288),
    ("e4m3", 2000, 570), ("e4m3", 2000, 1150), ("e4m3", 700, 800)])
def test_resident_groups_equal_streaming(gpu_ctx, kind, n, B):
    inst = _instance(kind, n)
    got = _run(gpu_ctx, inst, B, 11)
    ref = _run(gpu_ctx, inst, B, 11, (128, 0), streaming=True)
    assert (got[3]["resident"], ref[3]["resident"]) == (1, 0)
    _same(got, ref)
