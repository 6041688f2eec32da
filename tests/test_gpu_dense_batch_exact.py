"""Batched dense sketches in more tensors than the GPU holds blocks at once:
each tensor is summed by one block per group of sketches, in integers, and
rounded once.  With entries that are whole numbers below 2^25 the fixed-point
step divides them exactly, so every output is the exact sum rounded to FP32.
Needs a GPU."""
from __future__ import annotations

import numpy as np
import pytest

from gpu_common import cuda, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fcs():
    import paper_2106_13062_gb300 as m
    m.build()
    return m


@pytest.fixture(scope="module")
def ctx(fcs):
    c = fcs.Context()
    yield c
    c.close()


@pytest.mark.parametrize("shape,J,D,nb,bits", [
    # full last mode, one group of sketches: sums of 128 entries a bin
    ((512, 512), [1024, 1024], 10, 170, 22),
    # two groups of sketches, two leading modes; sums of 7 entries a bin
    ((16, 16, 256), [3000, 3000, 3000], 10, 170, 24),
    # three leading modes, a last mode with empty lanes
    ((4, 8, 16, 100), [300, 200, 400, 150], 4, 700, 22),
])
def test_one_rounding(fcs, ctx, orc, shape, J, D, nb, bits):
    g = np.random.default_rng(701)
    T = g.integers(-(1 << bits) + 1, 1 << bits, (nb,) + shape).astype(np.float32)
    ho, so = orc.make_hashes(702, list(shape), J, D)
    got = host(fcs.fcs_sketch_dense(ctx, cuda(T), J, cuda(ho), cuda(so), batched=True))
    Jt = sum(J) - len(J) + 1
    off = np.cumsum([0, *shape])
    rounded = 0
    for d in range(D):
        bins, sign = np.zeros(1, np.int64), np.ones(1, np.int64)
        for n, i in enumerate(shape):
            hn = ho[d, off[n]:off[n] + i].astype(np.int64)
            sn = so[d, off[n]:off[n] + i].astype(np.int64)
            bins, sign = (bins[:, None] + hn).ravel(), (sign[:, None] * sn).ravel()
        for b in {0, 1, nb // 2, nb // 2 + 1, nb - 2, nb - 1}:
            # whole numbers below 2^53: exact in FP64, in any order
            ref = np.bincount(bins, weights=T[b].ravel().astype(np.float64) * sign, minlength=Jt)
            rounded += int((ref != ref.astype(np.float32)).sum())
            np.testing.assert_array_equal(got[b, d], ref.astype(np.float32))
    assert rounded > 100                    # sums that FP32 does not hold
