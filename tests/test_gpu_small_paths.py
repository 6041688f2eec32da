"""Kernels for small work against the FP64 oracle or FP64 numpy at the sizes
where they can go wrong: dense sketches of small tensors (one block per
tensor), inner products of few sketches, and the ALS update at every rank
class.  Needs a GPU."""
from __future__ import annotations

import numpy as np
import pytest

import synth
from gpu_common import CONTRACT_RTOL, assert_sketch_close, cuda, host

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


def _dense_ref(orc, T, J, ho, so):
    return np.stack([orc.fcs_dense(t.astype(np.float64), J, ho, so) for t in T])


@pytest.mark.parametrize("shape,J,D,nb", [
    ((1,), [1], 1, 1), ((7, 7, 32), [60, 60, 60], 5, 400), ((3, 5, 7), [4, 9, 11], 3, 1),
    ((2, 1, 3, 1, 2), [3, 2, 5, 1, 4], 16, 5), ((8192,), [300], 4, 200), ((91, 90), [50, 70], 2, 160),
    ((8193,), [3000], 1, 160), ((33, 31), [16384, 16384], 1, 160), ((64, 64), [90, 80], 1, 3),
])
@pytest.mark.parametrize("kind", ["normal", "spike", "tiny", "huge"])
def test_dense_small_tensors(fcs, ctx, orc, shape, J, D, nb, kind):
    T = synth.gaussian(401, (nb,) + shape)
    if kind == "spike":
        T.reshape(nb, -1)[0, 0] = 3e7
    elif kind != "normal":
        T = (T.astype(np.float64) * (1e-30 if kind == "tiny" else 1e30)).astype(np.float32)
    ho, so = orc.make_hashes(402, list(shape), J, D)
    got = host(fcs.fcs_sketch_dense(ctx, cuda(T), J, cuda(ho), cuda(so), batched=True))
    ref = _dense_ref(orc, T, J, ho, so)
    assert_sketch_close(got, ref)
    if kind == "spike":                  # the other bins keep their own accuracy
        S = np.zeros_like(T[0])
        S.reshape(-1)[0] = T.reshape(nb, -1)[0, 0]
        keep = orc.fcs_dense(S.astype(np.float64), J, ho, so) == 0
        for d in range(D):
            r = ref[0, d][keep[d]]
            if np.linalg.norm(r) > 0:
                assert np.linalg.norm(got[0, d][keep[d]] - r) <= 1e-5 * np.linalg.norm(r)


def test_dense_small_tensor_nan_and_bad_hash(fcs, ctx, orc):
    shape, J, D = (9, 10, 12), [20, 30, 40], 3
    T = synth.gaussian(403, (2,) + shape)
    T[1, 4, 4, 4], T[1, 2, 3, 5] = np.nan, np.inf
    ho, so = orc.make_hashes(404, list(shape), J, D)
    bad = ho.copy()
    bad[0, 3], bad[1, 9 + 2], bad[2, 19 + 7] = -1, 30, 1 << 29
    ref = _dense_ref(orc, T, J, ho, so)
    for d, (n, i) in enumerate([(0, 3), (1, 2), (2, 7)]):
        Z = T.copy()
        Z[(slice(None), *[slice(None)] * n, i)] = 0.0
        ref[:, d] = _dense_ref(orc, Z, J, ho, so)[:, d]
    got = host(fcs.fcs_sketch_dense(ctx, cuda(T), J, cuda(bad), cuda(so), batched=True))
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    fin = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), fin)
    assert np.linalg.norm(got[fin] - ref[fin]) <= 1e-5 * np.linalg.norm(ref[fin])


@pytest.mark.parametrize("shape,J,D,nb", [
    ((20, 16, 260), [90, 80, 300], 2, 33), ((12, 260), [50, 400], 3, 640), ((400,), [300], 1, 20000),
    ((4, 2, 3, 2, 2, 96), [9, 5, 7, 3, 4, 50], 2, 160), ((16, 16, 64), [3000, 3000, 3000], 10, 100),
])
@pytest.mark.parametrize("kind", ["normal", "spike", "nan"])
def test_dense_batch_rows(fcs, ctx, orc, shape, J, D, nb, kind):
    """Batches whose rows are shared out evenly over the CTAs, so that a CTA
    takes parts of several tensors: a large value or a NaN stays in its own."""
    T = synth.gaussian(411, (nb,) + shape)
    if kind != "normal":
        T.reshape(nb, -1)[nb // 2, 0] = 3e9 if kind == "spike" else np.nan
    ho, so = orc.make_hashes(412, list(shape), J, D)
    got = host(fcs.fcs_sketch_dense(ctx, cuda(T), J, cuda(ho), cuda(so), batched=True))
    pick = sorted({0, 1, nb // 2 - 1, nb // 2, nb // 2 + 1, nb - 1})
    ref = _dense_ref(orc, T[pick], J, ho, so)
    fin = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got[pick]), fin)
    assert np.isfinite(got).sum() == got.size - (~fin).sum()
    for g, r, f in zip(got[pick], ref, fin):
        assert np.linalg.norm(g[f] - r[f]) <= 1e-5 * np.linalg.norm(r[f])


@pytest.mark.parametrize("B,C,D,Jt", [(1, 1, 1, 1), (5, 3, 16, 31), (256, 10, 5, 178), (6, 130, 2, 33),
                                      (700, 9, 3, 1000), (2000, 200, 2, 40)])
def test_inner_products(fcs, ctx, B, C, D, Jt):
    sa, sw = synth.gaussian(405, (B, D, Jt)), synth.gaussian(406, (C, D, Jt))
    bias = synth.gaussian(407, (C,))
    y, raw = fcs.fcs_sketch_inner(ctx, cuda(sa), cuda(sw), cuda(bias), raw=True)
    ref = np.einsum("bdj,cdj->bcd", sa.astype(np.float64), sw.astype(np.float64))
    tol = CONTRACT_RTOL * np.linalg.norm(sa, axis=2)[:, None, :] * np.linalg.norm(sw, axis=2)[None]
    assert np.all(np.abs(host(raw) - ref) <= tol)
    assert np.all(np.abs(host(y) - (np.median(ref, axis=2) + bias)) <= tol.max(axis=2) + 1e-6)
    y2 = fcs.fcs_sketch_inner(ctx, cuda(sa), cuda(sw))
    assert np.all(np.abs(host(y2) - np.median(ref, axis=2)) <= tol.max(axis=2))


@pytest.mark.parametrize("R", [1, 2, 8, 9, 16, 17, 32])
def test_als_update_ranks(fcs, ctx, orc, R):
    """One sweep from orthogonal-ish factors: same factors as the oracle's
    loop (cond(G) stays below 10, so the contraction bar carries over)."""
    import oracle.algorithms as alg
    I, J, D = [90, 70, 110], [3000, 2000, 2500], 3
    U, lam = synth.cp_factors(408, I, R)
    ho, so = orc.make_hashes(409, I, J, D)
    hg, sg = cuda(ho), cuda(so)
    fT = fcs.fcs_sketch_cp(ctx, [cuda(u) for u in U], cuda(lam), J, hg, sg)
    init = [synth.orthonormal_columns(410 + n, i, R).T.astype(np.float32).copy() for n, i in enumerate(I)]
    F = [cuda(x.copy()) for x in init]
    lam_g = host(fcs.fcs_als(ctx, fT, I, J, hg, sg, F, 1))
    Fref, lref = alg.als(host(fT).astype(np.float64), I, J, ho, so, R, 1, init)
    np.testing.assert_allclose(lam_g, lref, rtol=3e-3)
    for f, fr in zip(F, Fref):
        np.testing.assert_allclose(host(f), fr, atol=3e-3)


@pytest.mark.parametrize("kind", ["all", "free", "both"])
@pytest.mark.parametrize("I,J,D,B,m", [
    ([300], [8192], 2, 3, 0), ([300], [16384], 1, 160, 0), ([40, 700], [4097, 4097], 3, 55, 1),
    ([50, 60, 70], [2049, 2900, 3000], 4, 5, 0), ([50, 60, 70], [5461, 5462, 5461], 2, 80, 2),
    ([30, 20, 25, 35], [3000, 2500, 100, 2600], 5, 2, 1), ([1200, 20], [9000, 7000], 1, 155, 0),
    ([30, 20, 25, 35], [4000, 2500, 100, 2600], 4, 40, 1), ([60, 90], [8000, 8385], 2, 3, 0),
])
def test_contract_long(fcs, ctx, orc, I, J, D, B, m, kind):
    """P = 8192 and 16384 at the ends of their ranges, every kind, in few and
    in more items than SMs (the row-pair engine at P = 16384), against the
    FP64 contraction of the same sketch."""
    if kind == "free" and len(I) == 1:
        pytest.skip("needs a vector to give the batch size")
    ho, so = orc.make_hashes(420, I, J, D)
    fT = synth.gaussian(421, (D, sum(J) - len(J) + 1))
    v = [synth.unit_vectors(422 + n, B, i) for n, i in enumerate(I)]
    hg, sg, fg, vg = cuda(ho), cuda(so), cuda(fT), [cuda(x) for x in v]
    f64, v64 = fT.astype(np.float64), [x.astype(np.float64) for x in v]
    ra = rf = None
    if kind == "both":
        _, _, ra, rf = fcs.fcs_contract_both(ctx, fg, vg, I, J, hg, sg, free_mode=m, raw=True)
    elif kind == "all":
        _, ra = fcs.fcs_contract(ctx, fcs.FCS_CONTRACT_ALL, fg, vg, I, J, hg, sg, raw=True)
    else:
        med, rf = fcs.fcs_contract(ctx, fcs.FCS_CONTRACT_FREE, fg, vg, I, J, hg, sg, free_mode=m,
                                   raw=True)
    for b in range(B):
        vb = [x[b] for x in v64]
        if ra is not None:
            ref = orc.contract_all(f64, vb, J, ho, so)
            scale = np.linalg.norm(f64, axis=1)
            assert np.all(np.abs(host(ra)[b] - ref) <= CONTRACT_RTOL * scale)
        if rf is not None:
            ref = orc.contract_free(f64, vb, m, J, ho, so)
            err = np.linalg.norm(host(rf)[b] - ref, axis=1)
            assert np.all(err <= CONTRACT_RTOL * np.linalg.norm(ref, axis=1))
