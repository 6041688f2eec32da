"""CP-ALS where its update can go wrong: factor matrices that share one buffer,
and solutions too large for shared memory.  Needs a GPU."""
from __future__ import annotations

import numpy as np
import pytest

import synth
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


def _problem(fcs, ctx, orc, I, J, D, R, seed):
    U, lam = synth.cp_factors(seed, I, R)
    ho, so = orc.make_hashes(seed + 1, I, J, D)
    hg, sg = cuda(ho), cuda(so)
    fT = fcs.fcs_sketch_cp(ctx, [cuda(u) for u in U], cuda(lam), J, hg, sg)
    init = [synth.orthonormal_columns(seed + 2 + n, i, R).T.astype(np.float32).copy()
            for n, i in enumerate(I)]
    return ho, so, hg, sg, fT, init


@pytest.mark.parametrize("share", [(0, 1), (1, 2), (0, 2), (0, 1, 2)])
def test_shared_factor_buffer(fcs, ctx, orc, share):
    """Modes that hold the same buffer see each other's updates at once, in
    the products of Gram matrices as in the contractions.  (cond(G) < 2 in
    the oracle's sweeps: the bar of the other ALS tests.)"""
    import oracle.algorithms as alg
    I, J, D, R = [40] * 3, [2000, 1500, 1800], 3, 6
    ho, so, hg, sg, fT, init = _problem(fcs, ctx, orc, I, J, D, R, 508)
    X = [x.astype(np.float64) for x in init]
    F = [cuda(x) for x in init]
    for n in share[1:]:
        X[n], F[n] = X[share[0]], F[share[0]]
    f64 = host(fT).astype(np.float64)
    for _ in range(2):
        for m in range(3):
            Mt = np.stack([alg.median(alg.contract_free(f64, [None if n == m else X[n][r]
                                                              for n in range(3)], m, J, ho, so,
                                                        I=I)) for r in range(R)])
            G = np.ones((R, R))
            for n in range(3):
                if n != m:
                    G *= X[n] @ X[n].T
            assert np.linalg.cond(G) < 2
            Y = np.linalg.solve(G, Mt)
            lref = np.linalg.norm(Y, axis=1)
            X[m][...] = Y / lref[:, None]
    lam = host(fcs.fcs_als(ctx, fT, I, J, hg, sg, F, 2))
    np.testing.assert_allclose(lam, lref, rtol=3e-3)
    for f, x in zip(F, X):
        np.testing.assert_allclose(host(f), x, atol=3e-3)


def test_solutions_of_both_sizes(fcs, ctx, orc):
    """R I_m on both sides of what shared memory holds (40 KiB), two sweeps,
    so that each kind's Gram matrices serve the other's update."""
    import oracle.algorithms as alg
    I, J, D, R = [700, 330, 90], [3000, 2000, 2500], 3, 32
    ho, so, hg, sg, fT, init = _problem(fcs, ctx, orc, I, J, D, R, 528)
    F = [cuda(x) for x in init]
    lam = host(fcs.fcs_als(ctx, fT, I, J, hg, sg, F, 2))
    Fref, lref = alg.als(host(fT).astype(np.float64), I, J, ho, so, R, 2, init)
    np.testing.assert_allclose(lam, lref, rtol=3e-3)
    for f, fr in zip(F, Fref):
        np.testing.assert_allclose(host(f), fr, atol=3e-3)
