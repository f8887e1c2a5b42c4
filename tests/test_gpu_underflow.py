"""Entries of x that underflow to 0 although they survive the operator (|w_i| / ||w||_2 below FP32's smallest
number): the support list keeps a place for each of them, as the count of survivors does, so that what reads
the list up to that count finds entries of this sweep, and the reported support holds the nonzeros of x."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [(4, 1500), (200, 9000)])
@pytest.mark.parametrize("form,s,kw", [(1, 700, {}), (2, 650, {}), (5, 1, dict(gamma=0.0)), (8, 1, dict(gamma=0.0)),
                                       (7, 620, dict(gamma_target=True, calib=9)), (1, 5, {})])
def test_survivors_that_underflow(n, p, form, s, kw):
    from paper_1212_4137_gb300 import build, spca
    build.build()
    spca.load()
    A = np.full((n, p), 1e-30, np.float32)
    A[:, 5] = 1e18 / np.sqrt(n)
    A[:, 900] = -1e17 / np.sqrt(n)
    h = spca.Handle(A)
    G = np.random.default_rng(n).uniform(0.5, 1.0, (3, p)).astype(np.float32)
    for engine in (spca.SPCA_ENGINE_SIMT, spca.SPCA_ENGINE_TC, spca.SPCA_ENGINE_AUTO):
        out = h.solve(form, 3, s=float(s), max_iter=4, tol=-1, x0=G, engine=engine, want_starts=True, **kw)
        X = out["start_x"].astype(np.float64)
        assert np.array_equal(out["support"], [5, 900]) and out["nnz"] == 2
        assert ((X != 0).sum(axis=1) == 2).all() and (np.abs(np.linalg.norm(X, axis=1) - 1.0) < 1e-6).all()
        U = X @ A.astype(np.float64).T
        want = np.abs(U).sum(axis=1) if form % 2 == 0 else (U ** 2).sum(axis=1)
        assert (np.abs(out["start_explained"] - want) <= 1e-6 * want).all()
    h.close()
