"""The x-step at the edges of its paths, against the FP64 oracle's operator: v shorter than a warp, at
the length of its list (1024), around the lengths where the CTA size changes, rows of every alignment;
ties at the threshold, zero rows, entries crowded into one index segment (the list overflows: full
pass), supports near and past the list's length, lambda_s = 0.  The bars are those of
test_gpu_parity.test_xstep_matches_oracle: identical supports, x within 1e-6, F and thresholds within
1e-6 relative (F of the L0 penalty relative to the size of its two terms)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1212_4137_gb300 import build, spca
    build.build()
    spca.load()
    return spca


def _rows(p, rng):
    V = rng.standard_normal((8, p)).astype(np.float32) * 3
    V[1, ::3] = 0.0
    V[2] = np.float32(0.75) * np.sign(V[2])                  # every magnitude equal
    V[3] = 0.0
    V[4, p // 2:p // 2 + max(1, p // 12)] *= 20              # crowded into one segment
    V[5] = np.round(V[5] * 4) / 4                            # many ties
    V[6] *= np.exp(rng.uniform(-12, 0, p)).astype(np.float32)   # many magnitudes
    V[7, -1] = 50.0
    return V


@pytest.mark.parametrize("p,pad,copies", [(1, 0, 1), (31, 1, 1), (64, 2, 1), (65, 3, 1), (1023, 1, 1), (1024, 0, 60),
                                          (1025, 2, 1), (2049, 3, 20), (8193, 1, 1), (16385, 0, 30), (32771, 2, 1),
                                          (52001, 1, 1)])
@pytest.mark.parametrize("form", range(1, 9))
def test_xstep_edges(lib, oracle, form, p, pad, copies):
    import torch
    rng = np.random.default_rng(17 * form + p)
    rows = _rows(p, rng)
    V = np.tile(rows, (copies, 1))                           # copies: more starts, smaller CTAs
    r, ld = V.shape[0], p + pad
    h = lib.Handle(np.zeros((2, p), np.float32))
    Vd = torch.zeros((r, ld), dtype=torch.float32, device="cuda")
    Vd[:, :p] = torch.from_numpy(V).cuda()
    Xd = torch.full((r, ld), np.nan, dtype=torch.float32, device="cuda")
    Fd = torch.zeros(r, dtype=torch.float64, device="cuda")
    Nd = torch.zeros(r, dtype=torch.int32, device="cuda")
    Td = torch.zeros(r, dtype=torch.float64, device="cuda")
    for s in sorted({1, min(p, 7), min(p, 599), min(p, 601), p}):
        for calibrate in ((False, True) if form >= 5 else (False,)):
            gamma = 2.0 if form >= 5 and not calibrate else 0.0
            st = lib.spca_xstep(h.h, form, float(s), gamma, calibrate, Vd.data_ptr(), ld, r, Xd.data_ptr(), ld,
                                Fd.data_ptr(), Nd.data_ptr(), Td.data_ptr())
            assert st == 0, lib.spca_last_error(h.h)
            X, F, N, T = Xd[:, :p].cpu().numpy(), Fd.cpu().numpy(), Nd.cpu().numpy(), Td.cpu().numpy()
            for k in range(1, copies):                       # every copy of a row gives the same bits
                for a in (X, F, N, T):
                    np.testing.assert_array_equal(a[8 * k:8 * k + 8], a[:8])
            for c in range(8):
                v = rows[c].astype(np.float64)
                ref = oracle.xstep(form, v, float(s), gamma, calibrate)
                if form in (3, 4) and s < p:
                    # entries within FP32 rounding of lambda_s may go either way, and where all
                    # magnitudes are equal lambda_s is their size or 0: x is then checked by its norm
                    m = np.abs(v)
                    if np.any(np.abs(m - ref.thr) <= 1e-6 * max(ref.thr, 1e-30)) or len(np.unique(m[m > 0])) <= 1:
                        continue
                assert N[c] == ref.nnz, (c, s, calibrate, N[c], ref.nnz)
                np.testing.assert_array_equal(X[c] != 0, ref.x != 0)
                assert np.abs(X[c] - ref.x).max() < 1e-6, (c, s, calibrate)
                scale = max(1.0, abs(ref.F), ref.thr * ref.nnz if form in (5, 6) else 0.0)
                assert abs(F[c] - ref.F) <= 1e-6 * scale, (c, s, calibrate, F[c], ref.F)
                assert abs(T[c] - ref.thr) <= 1e-6 * max(1.0, abs(ref.thr)), (c, s, calibrate, T[c], ref.thr)
    h.close()
