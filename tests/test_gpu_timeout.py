"""timeout_us in the one-launch solve of small problems: the sweeps then run in launches of four, so a solve with
a large max_iter ends soon after its limit, and one that stays within it gives the bits that it gives without a
limit (a start goes on from its support list and state, at any number of sweeps and any support)."""
import time

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


@pytest.mark.parametrize("n,p,r", [(60, 300, 3), (100, 900, 20), (900, 1000, 1), (900, 1000, 16)])
def test_small_solve_ends_at_its_limit(lib, n, p, r):
    h = lib.Handle(np.random.default_rng(n).standard_normal((n, p)).astype(np.float32))
    kw = dict(s=10.0, tol=-1, seed=1)
    good = h.solve(1, r, max_iter=6, **kw)
    t = time.perf_counter()
    with pytest.raises(lib.SpcaError) as e:
        h.solve(1, r, max_iter=1_000_000, timeout_us=20_000, **kw)
    assert e.value.status == lib.SPCA_E_TIMEOUT
    assert time.perf_counter() - t < 2.0      # (all of its sweeps would take five seconds and more)
    assert np.array_equal(h.solve(1, r, max_iter=6, **kw)["x"], good["x"])
    h.close()


@pytest.mark.parametrize("n,p,r", [(30, 200, 17), (100, 500, 40), (700, 1000, 4), (64, 2048, 3)])
def test_a_limit_does_not_change_the_bits(lib, n, p, r):
    A = I.spiked_matrix(n, p, I.spiked_thetas(n, p), 12, n + p, dtype=np.float32)
    A[:, 3] = 0.0
    G = np.random.default_rng(p).standard_normal((r, p)).astype(np.float32)
    G[1] = 0.0
    G[2 % r] = 0.0
    G[2 % r, 3] = 1.0
    h = lib.Handle(A)
    cases = [(form, s, kw, it, tol) for form, s, kw in
             ((1, 7, {}), (2, p, {}), (3, p // 3, {}), (4, 9, {}), (6, 1, dict(gamma=0.5)), (5, 11, dict(gamma_target=True, calib=5)),
              (7, 11, dict(gamma_target=True, calib=3)), (8, 1, dict(gamma=1e-7)))
             for it, tol in ((1, -1), (3, -1), (4, -1), (5, -1), (9, -1), (60, 1e-6))]
    for form, s, kw, it, tol in cases:
        a, b = (h.solve(form, r, s=float(s), max_iter=it, tol=tol, x0=G, want_starts=True, timeout_us=limit, **kw)
                for limit in (0, 60_000_000))
        for k in ("start_x", "start_F", "start_gamma", "start_iters", "start_status", "start_objective", "x", "y",
                  "support"):
            assert np.array_equal(a[k], b[k]), (form, s, it, tol, k)
        assert a["best_start"] == b["best_start"] and a["sweeps_total"] == b["sweeps_total"]
    bad = G.copy()
    bad[0, p // 2] = np.inf
    with pytest.raises(lib.SpcaError) as e:
        h.solve(1, r, s=7.0, max_iter=50, tol=-1, x0=bad, timeout_us=60_000_000)
    assert e.value.status == lib.SPCA_E_INVALID
    h.close()
