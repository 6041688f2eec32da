"""Dense sketches of small tensors whose entries differ widely in size: one
rounding per output, as for entries of one size.  The entries are whole
numbers, the small ones up to 1000 and a twentieth of them near 2^24, so the
exact sums are known and most do not fit FP32.  Needs a GPU."""
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


@pytest.mark.parametrize("shape,J,D,nb", [((64, 64), [90, 80], 5, 160), ((8192,), [300], 1, 200),
                                          ((9, 7, 11), [20, 30, 40], 16, 160)])
def test_one_rounding(fcs, orc, shape, J, D, nb):
    ctx = fcs.Context()
    g = np.random.default_rng(711)
    small = g.integers(-1000, 1001, (nb,) + shape)
    large = g.integers(1 << 23, 1 << 24, small.shape) * g.choice([-1, 1], small.shape)
    T = np.where(g.random(small.shape) < 0.05, large, small).astype(np.float32)
    ho, so = orc.make_hashes(712, list(shape), J, D)
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
        for b in (0, 1, nb - 1):
            ref = np.bincount(bins, weights=T[b].ravel().astype(np.float64) * sign, minlength=Jt)
            rounded += int((ref != ref.astype(np.float32)).sum())
            np.testing.assert_array_equal(got[b, d], ref.astype(np.float32))
    assert rounded > 0
    ctx.close()
