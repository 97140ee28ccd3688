"""FP64 couplings in the integer forms of the energy kernel: rounding them to
one scale may cost no more than rounding each to FP64 would."""

import numpy as np
import pytest

import synth
from oracle import ising
from paper_2312_05837_gb300 import api

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def _instance(n, below, bits=50):
    """Equal couplings `below` binary orders under the largest one, their last
    bit worth half a unit of a scale of 58 bits (or less): with equal spins
    every rounding to a coarser scale has the same sign."""
    J = np.full((n, n), 2.0 ** -below * (1.0 + 2.0 ** -(bits - 1)))
    J[0, 1] = J[1, 0] = 1.0
    np.fill_diagonal(J, 0.0)
    return synth.Instance(n=n, layout="dense", J=J, name="steps")


def _ordered(J, s):
    """s^T J s as a warp per row and vector adds it: every 32nd column per lane, an
    xor tree, eight rows per warp, eight warps per block, the blocks' partials
    32 at a time and an xor tree (products by +-1 are exact)."""
    def tree(x):
        for o in (16, 8, 4, 2, 1):
            x = x + x[..., np.arange(32) ^ o]
        return x[..., 0]

    def fold(x):
        a = np.zeros(x.shape[:-1])
        for k in range(x.shape[-1]):
            a = a + x[..., k]
        return a
    n = len(s)
    p = np.pad(J * s, ((0, 0), (0, -n % 32))).reshape(n, -1, 32)
    rows = tree(fold(np.moveaxis(p, 1, 2))) * s
    blocks = fold(fold(np.pad(rows, (0, -n % 64)).reshape(-1, 8, 8)))
    parts = np.pad(blocks, (0, -len(blocks) % 32)).reshape(-1, 32)
    return tree(fold(parts.T))


# binary orders below the largest coupling: inside and outside every scale's range
@pytest.mark.parametrize("below", [2, 5, 6, 7, 8, 9, 10, 11])
@pytest.mark.parametrize("n,count", [(40, 3), (200, 1), (200, 5), (1030, 4), (2050, 2), (1030, 260)])
def test_no_further_off_than_an_fp64_sum(gpu_ctx, below, n, count):
    inst = _instance(n, below)
    s = np.ones((count, n), np.int8)
    s[1::2, 1::7] = -1
    cq, _ = ising.coefficients(inst.j_scale, inst.convention)
    pick = list(range(min(count, 2)))
    E = api.energy(gpu_ctx, inst, s)
    total = float(np.abs(inst.J).sum())
    for k in pick:
        x = s[k].astype(np.longdouble)
        ref = ((inst.J.astype(np.longdouble) @ x) * x).sum()
        off = abs(float(_ordered(inst.J, s[k].astype(np.float64)) - ref))
        # the FP64 sum's own error, or the couplings' roundings (2^-53 sum |J|), and
        # three roundings of the result
        assert abs(float(E[k] / np.longdouble(cq) - ref)) <= off + 4 * EPS * total
