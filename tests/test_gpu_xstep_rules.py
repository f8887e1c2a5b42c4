"""spca_xstep on both sides of each line of its dispatch, against the FP64 oracle's operator with the bars of
test_gpu_xstep_edges (identical supports, x within 1e-6, F and thresholds within 1e-6 relative), and the
launches that each side takes: the list, or the full pass of every start in one launch where the list does
not pay (few entries of v per selected one, more selected entries than a list holds, lambda_s with s above
150, s = p).  Values: noise with entries that stand out, and heavy tails, whose active set outgrows the list
of some starts and not of others; fixed thresholds that one segment of v alone outgrows, or just does not."""
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


def _values(p, rng):
    v = rng.standard_normal((6, p)) * 3
    v[1, ::97] *= 2.5
    v[2] = rng.standard_t(2, p)
    v[3] = rng.standard_normal(p) / np.maximum(np.abs(rng.standard_normal(p)) + np.abs(rng.standard_normal(p)), 1e-3)
    v[4, rng.choice(p, max(1, p // 40), replace=False)] *= 30
    v[5] *= np.exp(rng.uniform(-6, 0, p))
    return v.astype(np.float32)


def _check(lib, oracle, p, copies, form, s, calibrate, gamma, launches, V=None):
    import torch
    rows = _values(p, np.random.default_rng(p + form)) if V is None else V
    k = rows.shape[0]
    r = k * copies
    h = lib.Handle(np.zeros((2, p), np.float32))
    Vd = torch.from_numpy(np.tile(rows, (copies, 1))).cuda()
    Xd = torch.full((r, p), np.nan, dtype=torch.float32, device="cuda")
    Fd, Td = (torch.zeros(r, dtype=torch.float64, device="cuda") for _ in range(2))
    Nd = torch.zeros(r, dtype=torch.int32, device="cuda")
    before = h.profile_query(lib.SPCA_K_XSTEP)[0]
    st = lib.spca_xstep(h.h, form, float(s), gamma, calibrate, Vd.data_ptr(), p, r, Xd.data_ptr(), p, Fd.data_ptr(),
                        Nd.data_ptr(), Td.data_ptr())
    assert st == 0, lib.spca_last_error(h.h)
    assert h.profile_query(lib.SPCA_K_XSTEP)[0] - before == launches
    X, F, N, T = Xd.cpu().numpy(), Fd.cpu().numpy(), Nd.cpu().numpy(), Td.cpu().numpy()
    h.close()
    for q in range(1, copies):
        for a in (X, F, N, T):
            np.testing.assert_array_equal(a[k * q:k * q + k], a[:k])
    for c in range(k):
        ref = oracle.xstep(form, rows[c].astype(np.float64), float(s), gamma, calibrate)
        m = np.abs(rows[c].astype(np.float64))
        if form in (3, 4) and np.any(np.abs(m - ref.thr) <= 1e-6 * max(ref.thr, 1e-30)):
            continue                                         # an entry within FP32 rounding of lambda_s
        assert N[c] == ref.nnz, (c, N[c], ref.nnz)
        np.testing.assert_array_equal(X[c] != 0, ref.x != 0)
        assert np.abs(X[c] - ref.x).max() < 1e-6, c
        scale = max(1.0, abs(ref.F), ref.thr * ref.nnz if form in (5, 6) else 0.0)
        assert abs(F[c] - ref.F) <= 1e-6 * scale, (c, F[c], ref.F)
        assert abs(T[c] - ref.thr) <= 1e-6 * max(1.0, abs(ref.thr)), (c, T[c], ref.thr)


# (p, copies of 6 rows, s, launches): a 25th of v up to two starts per SM (6 x 50 = 300), a 13th above
# (6 x 51 = 306); at most 500 entries; past an SM for each start the full pass of long rows is a second launch
@pytest.mark.parametrize("p,copies,s,launches", [(2500, 1, 100, 1), (2499, 1, 100, 1), (2500, 50, 101, 1),
                                                 (2500, 51, 101, 1), (1300, 51, 100, 1), (1299, 51, 100, 1),
                                                 (20011, 1, 500, 1), (20011, 1, 501, 1), (20011, 60, 500, 2),
                                                 (20011, 60, 501, 1), (20011, 60, 450, 2), (20011, 1, 20011, 1),
                                                 (300, 1, 12, 1), (300, 1, 13, 1), (70, 1, 60, 1), (60, 60, 40, 1)])
@pytest.mark.parametrize("form,calibrate", [(1, 0), (6, 1), (7, 1)])
def test_selections(lib, oracle, p, copies, s, launches, form, calibrate):
    _check(lib, oracle, p, copies, form, s - calibrate if s < p else p, calibrate, 0.0, launches)


@pytest.mark.parametrize("p,copies,s,launches", [(3000, 1, 150, 1), (3000, 1, 151, 1), (3000, 60, 150, 1),
                                                 (20011, 1, 50, 1), (20011, 1, 150, 1), (20011, 60, 150, 2),
                                                 (20011, 60, 151, 1), (60001, 1, 100, 1), (20011, 60, 20, 2),
                                                 (500, 1, 140, 1), (500, 60, 480, 1)])
@pytest.mark.parametrize("form", [3, 4])
def test_lambda(lib, oracle, p, copies, s, launches, form):
    _check(lib, oracle, p, copies, form, s, 0, 0.0, launches)


# fixed thresholds: 63, 64 and 65 entries above in the first segment, or in another one, or everywhere
@pytest.mark.parametrize("copies,launches", [(1, 1), (45, 2)])
@pytest.mark.parametrize("form", [5, 8])
def test_fixed_threshold(lib, oracle, copies, launches, form):
    p = 20011
    rng = np.random.default_rng(form)
    V = rng.uniform(-0.9, 0.9, (7, p)).astype(np.float32)
    seg = ((p + 15) // 16 + 127) // 128 * 128
    for row, (at, n) in enumerate([(0, 63), (0, 64), (0, 65), (5 * seg, 65), (0, 1200)]):
        V[row, at + rng.choice(seg, min(n, seg), replace=False)] = rng.uniform(1.1, 3.0, min(n, seg))
    V[5] *= 5
    _check(lib, oracle, p, copies, form, 1, 0, 1.0, launches, V)
