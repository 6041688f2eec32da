"""The row-pair FFT engine of the CP route (P = 8192, 16384, 32768) at the
edges of its ranges, against the FP64 oracle: every input pruning of the row
step on both sides of its limit, columns longer than the prefetch, more ranks
than resident blocks, and the shared-memory limits (blocks per SM, the longest
hash range at P = 32768).  Needs a GPU."""
from __future__ import annotations

import numpy as np
import pytest

import synth
from gpu_common import assert_sketch_close, cuda, host

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


def _case(fcs, orc, I, J, R, D, seed):
    U, lam = synth.cp_factors(seed, I, R)
    ho, so = orc.make_hashes(seed + 1, I, J, D)
    ref = orc.fcs_cp([u.astype(np.float64) for u in U], lam.astype(np.float64), J, ho, so)
    return [cuda(u) for u in U], cuda(lam), cuda(ho), cuda(so), ref


@pytest.mark.parametrize("I,J,R,D", [
    # P = 8192: ra = J / 16 at 128 | 129, 176 | 177, 256 | 257, 512
    ([40, 30, 20], [2048, 2048, 2048], 3, 2),
    ([40, 30, 20], [2052, 2050, 2047], 3, 2),
    ([40, 30, 20], [2816, 2815, 1000], 3, 2),
    ([40, 30], [2820, 2700], 3, 2),
    ([40, 30], [4096, 1000], 3, 2),
    ([40, 30], [4099, 1000], 3, 2),
    ([600, 1], [8191, 2], 3, 2),
    # P = 16384: ra = J / 32; a column longer than the prefetch
    ([40, 30, 20], [4096, 4096, 4096], 3, 2),
    ([40, 1100, 20], [4098, 4096, 100], 3, 2),
    ([40, 30], [5632, 5632], 3, 2),
    ([40, 30], [5635, 5000], 3, 2),
    ([40, 30], [8192, 1000], 3, 2),
    ([40, 30], [8257, 1000], 3, 2),
    # P = 32768: ra = J / 64
    ([40, 30, 20], [8192, 8192, 8192], 3, 2),
    ([40, 2200, 20], [8196, 8190, 500], 3, 2),
    ([40, 30], [11264, 11000], 3, 2),
    ([40, 30], [11269, 6000], 3, 2),
    ([40, 30], [16384, 1000], 3, 2),
    ([40, 30], [17984, 1000], 3, 2),
    ([40, 30], [17985, 1000], 3, 2),
])
def test_row_step_limits(fcs, ctx, orc, I, J, R, D):
    U, lam, h, s, ref = _case(fcs, orc, I, J, R, D, 301)
    assert_sketch_close(host(fcs.fcs_sketch_cp(ctx, U, lam, J, h, s)), ref)


@pytest.mark.parametrize("J", [5000, 9000, 17000])
def test_more_ranks_than_blocks(fcs, ctx, orc, J):
    """Order 1, R above the number of resident blocks: blocks take several
    ranks from the shared counter, twice in a row on one context."""
    U, lam, h, s, ref = _case(fcs, orc, [50], [J], 1300, 1, 311)
    for _ in range(2):
        assert_sketch_close(host(fcs.fcs_sketch_cp(ctx, U, lam, [J], h, s)), ref)


def test_batch_long_and_tall(fcs, ctx, orc):
    """A plan without a grain over P = 32768, P = 16384 and 8192 with scatter
    buffers that do and do not cost a resident block, and a hash range beyond
    the engine; with room for it, and with a budget that sends P = 32768 to
    the in-place route."""
    shapes = [([60, 50, 40], [7000, 7000, 7000], 9, 2), ([60, 50], [9000, 4000], 7, 3),
              ([60, 50, 40], [4000, 4000, 4000], 11, 2), ([60, 50], [6000, 1500], 5, 1),
              ([60, 50, 40], [2000, 2000, 2000], 6, 4), ([40, 30], [18000, 900], 2, 1)]
    data = [_case(fcs, orc, *sh, 320 + k) for k, sh in enumerate(shapes)]
    for budget in (None, 880 << 10):
        c = fcs.Context(budget=budget)
        probs, outs = [], []
        for (I, J, R, D), (U, lam, h, s, ref) in zip(shapes, data):
            pr, out = fcs.cp_problem(U, lam, J, h, s)
            probs.append(pr)
            outs.append(out)
        plan = fcs.BatchPlan(c, probs)
        for _ in range(2):
            plan.launch()
            for out, d in zip(outs, data):
                assert_sketch_close(host(out), d[4])
        grain, cls = plan.config()
        assert grain == 0 and [x[0] for x in cls] == [16384, 8192]
        c.close()
