"""Contractions at P = 16384 whose results lie near the top of FP32's range:
a batch of more items than SMs (the row-pair engine) stays finite wherever
batches of a few items do, and gives their results.  Needs a GPU."""
from __future__ import annotations

import numpy as np
import pytest

import synth
from gpu_common import CONTRACT_RTOL, cuda, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fcs():
    import paper_2106_13062_gb300 as m
    m.build()
    return m


@pytest.mark.parametrize("I,J,D,B,m", [([40, 50, 30], [5000, 5000, 5000], 5, 64, 0),
                                       ([30, 20, 25, 35], [4000, 3500, 2500, 2600], 4, 64, 3)])
def test_large_batch_has_the_range_of_a_small_one(fcs, orc, I, J, D, B, m):
    ctx = fcs.Context()
    ho, so = orc.make_hashes(801, I, J, D)
    hg, sg = cuda(ho), cuda(so)
    fT = synth.gaussian(802, (D, sum(J) - len(J) + 1))
    v = [synth.gaussian(803 + n, (B, i)) for n, i in enumerate(I)]
    few = 8
    top = None
    for e in range(90, 128):               # the largest scale at which few items stay finite
        f = cuda(fT * np.float32(2.0 ** e))
        parts = [fcs.fcs_contract_both(ctx, f, [cuda(x[k:k + few]) for x in v], I, J, hg, sg,
                                       free_mode=m) for k in range(0, B, few)]
        a, r = (np.concatenate([host(p[i]) for p in parts]) for i in (0, 1))
        if not (np.isfinite(a).all() and np.isfinite(r).all()):
            break
        top = (f, a, r)
    f, a, r = top
    got_a, got_r = (host(x) for x in
                    fcs.fcs_contract_both(ctx, f, [cuda(x) for x in v], I, J, hg, sg, free_mode=m))
    assert np.isfinite(got_a).all() and np.isfinite(got_r).all()
    # the two engines' errors together; T(v, .., v) on the scale of its inner product
    a, r, got_a, got_r = (x.astype(np.float64) for x in (a, r, got_a, got_r))
    scale = np.linalg.norm(host(f).astype(np.float64), axis=1).max() * np.prod(
        [np.linalg.norm(x.astype(np.float64), axis=1) for x in v], axis=0)
    assert np.all(np.abs(got_a - a) <= 2 * CONTRACT_RTOL * scale)
    assert np.all(np.linalg.norm(got_r - r, axis=1) <= 2 * CONTRACT_RTOL * np.linalg.norm(r, axis=1))
    ctx.close()
