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


def test_hash_ranges_are_part_of_the_shape(fcs):
    """P = 16384 with hash ranges that leave room for two resident blocks per
    SM and with one that does not; P = 32768 on and off the batch kernels: a
    shape tuned for one is not used for the other."""
    c = fcs.Context()
    for Ja, Jb in (([6500, 6500], [9000, 4000]), ([9000, 9000], [18000, 900])):
        I, R, D = [120, 90], 6, 2
        pa, _ka = _batch(fcs, c, [(I, Ja, R, D)], 911)
        pb, _kb = _batch(fcs, c, [(I, Jb, R, D)], 912)
        g = fcs.fcs_batch_autotune(c, pa)
        for probs, grain in ((pa, g), (pb, 0)):
            plan = fcs.BatchPlan(c, probs)
            assert plan.config()[0] == grain
            plan.close()
    c.close()


def _fnv(values):
    x = 1469598103934665603
    for v in values:
        for b in range(8):
            x = ((x ^ ((v >> (8 * b)) & 0xff)) * 1099511628211) & (2 ** 64 - 1)
    return x


def test_entries_of_earlier_kernels_are_not_used(fcs, monkeypatch, tmp_path):
    """A file written before the engines changed (the signature was the hash
    of the problem count and of (log2 M, N, D, R, max I_n)): read and kept,
    but its grain is not taken."""
    I, J, R, D = [120, 90], [6500, 6500], 6, 2
    path = tmp_path / "tune.txt"
    line = "%016x 4 13:1:2:1" % _fnv([1, 13, 2, D, R, max(I)])
    path.write_text(line + "\n")
    monkeypatch.setenv("FCS_AUTOTUNE_CACHE", str(path))
    c = fcs.Context()
    probs, _keep = _batch(fcs, c, [(I, J, R, D)], 921)
    plan = fcs.BatchPlan(c, probs)
    grain, cls = plan.config()
    assert grain == 0 and [(P, ipc) for P, _, ipc, _, _ in cls] == [(16384, 1)]
    plan.close()
    fcs.fcs_batch_autotune(c, probs)
    assert line in path.read_text().splitlines() and len(path.read_text().splitlines()) == 2
    c.close()
