"""Which solves of small problems take one launch: any support up to 2^17 entries of A; above, n times the
expected support up to 2^18 (s, 2 s for lambda_s, all of x for a fixed penalty).  Each side of the lines against
the FP64 oracle with the bars of test_gpu_paths; the one-launch solve makes no launch of v = A^T y."""
import numpy as np
import pytest

from paper_1212_4137_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1212_4137_gb300 import build, spca
    build.build()
    spca.load()
    return spca


@pytest.mark.parametrize("n,p,r,form,s,kw,one_launch", [
    (1000, 1000, 1, 1, 262, {}, True), (1000, 1000, 1, 1, 263, {}, False), (1000, 1000, 3, 2, 1000, {}, False),
    (1000, 1000, 2, 3, 131, {}, True), (1000, 1000, 2, 4, 132, {}, False),
    (512, 1024, 4, 6, 512, dict(gamma_target=True, calib=50), True),
    (512, 1024, 4, 7, 513, dict(gamma_target=True, calib=50), False),
    (200, 2000, 5, 5, 1, dict(gamma=2.0), False), (131, 2001, 5, 7, 1, dict(gamma=1.0), True),
    (128, 1024, 5, 1, 1024, {}, True), (128, 1024, 5, 8, 1, dict(gamma=0.5), True), (129, 1024, 2, 1, 1024, {}, True),
    (300, 1024, 2, 1, 1024, {}, False)])
def test_small_solve_route(lib, oracle, n, p, r, form, s, kw, one_launch):
    A = I.spiked_matrix(n, p, I.spiked_thetas(n, p), 12, n + p, dtype=np.float32)
    G = np.random.default_rng(s).standard_normal((r, p)).astype(np.float32)
    h = lib.Handle(A)
    before = h.profile_query(lib.SPCA_K_V)[0]
    out = h.solve(form, r, s=float(s), max_iter=3, tol=-1, x0=G, want_starts=True, **kw)
    assert (h.profile_query(lib.SPCA_K_V)[0] == before) == one_launch
    h.close()
    ref = oracle.solve(A.astype(np.float64), form, G.astype(np.float64), s=float(s), max_iter=3, tol=-1, **kw)
    assert np.array_equal(out["start_status"], ref.status) and np.array_equal(out["start_iters"], ref.iters)
    assert (np.abs(out["start_objective"] - ref.f) <= 1e-5 * np.maximum(1.0, np.abs(ref.f))).all()
    assert (np.abs(out["start_x"] - ref.X).max(axis=1) <= 1e-4).all()
