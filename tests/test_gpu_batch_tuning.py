"""What the batch autotuner returns, and for which batches its choice is used.
Needs a GPU."""
from __future__ import annotations

import pytest

import synth
from gpu_common import assert_sketch_close, cuda, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fcs():
    import paper_2106_13062_gb300 as m
    m.build()
    return m


def _batch(fcs, c, shapes, seed):
    probs, keep = [], []
    for k, (I, J, R, D) in enumerate(shapes):
        U, lam = synth.cp_factors(seed + k, I, R)
        Ug, lamg = [cuda(u) for u in U], cuda(lam)
        h, s = fcs.fcs_make_hashes(c, seed + 50 + k, I, J, D)
        pr, out = fcs.cp_problem(Ug, lamg, J, h, s)
        ref = host(fcs.fcs_sketch_cp(c, Ug, lamg, J, h, s))
        probs.append(pr)
        keep.append((Ug, lamg, h, s, out, ref))
    return probs, keep


def test_returned_grain(fcs, monkeypatch, tmp_path):
    """The grain is a number of ranks, also where a cut problem by problem is
    the fastest (ranks from 1 to 300 in one FFT length); the plan of the tuned
    batch names it and another context reads it from the file."""
    monkeypatch.setenv("FCS_AUTOTUNE_CACHE", str(tmp_path / "tune.txt"))
    c = fcs.Context()
    shapes = [([200, 150, 100], [1300, 1300, 1300], R, D)
              for R, D in ((300, 5), (1, 10), (150, 2), (7, 3), (260, 4), (30, 8))]
    probs, keep = _batch(fcs, c, shapes, 901)
    g = fcs.fcs_batch_autotune(c, probs)
    assert g in (1, 2, 4, 8, 16, 32, 64)
    c2 = fcs.Context()
    for ctx, grain in ((c, 0), (c, g), (c2, 0)):
        plan = fcs.BatchPlan(ctx, probs, grain=grain)
        assert plan.config()[0] == g
        plan.launch()
        for k in keep:
            assert_sketch_close(host(k[4]), k[5])
            k[4].zero_()
        plan.close()
    c2.close()
    c.close()
