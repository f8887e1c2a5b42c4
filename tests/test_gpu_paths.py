"""The rules that pick a kernel by size, at the sizes where they change: widths of the tensor-core tiles and
of the few-start products, the support gather's two shapes, the one-launch solve of small problems (CTAs per
start, columns of A in shared memory or not, its largest problem), the read-backs and the copy of a solve's
results, and the work items and column searches of a sparse A.

Bars, from before the first run: products relative to sum |a b| as test_gpu_products (2e-6 for FP32 FMA
chains of a few thousand terms, K/16 truncations of 2^-23 on the tensor cores) and test_gpu_sparse (2^-24 per
term of a chain); solves of 3 sweeps as test_gpu_parity (identical sweep counts and status, at least 95 % of
the starts with the objective within 1e-5 and x within 1e-4 of the FP64 oracle, best objective within 1e-5)."""
import numpy as np
import pytest
import scipy.sparse as sps

from paper_1212_4137_gb300 import inputs as I

pytestmark = pytest.mark.gpu
DEGENERATE = 2


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1212_4137_gb300 import build, spca
    build.build()
    spca.load()
    return spca


def _products(lib, h, form, engine, X):
    import torch
    r, p = X.shape
    Xd = torch.from_numpy(np.ascontiguousarray(X, np.float32)).cuda()
    Ud = torch.zeros((r, h.n + 1), dtype=torch.float32, device="cuda")
    Vd = torch.zeros((r, p + 3), dtype=torch.float32, device="cuda")
    st = lib.spca_products(h.h, form, engine, Xd.data_ptr(), p, r, Ud.data_ptr(), h.n + 1, Vd.data_ptr(), p + 3)
    assert st == 0, lib.spca_last_error(h.h)
    torch.cuda.synchronize()
    return Ud[:, :h.n].cpu().numpy().astype(np.float64), Vd[:, :p].cpu().numpy().astype(np.float64)


def _check_products(A64, X, U, V, form, bar_u, bar_v):
    X = X.astype(np.float64)
    ref, scale = (A64 @ X.T).T, (abs(A64) @ np.abs(X).T).T
    assert (np.abs(U - ref) <= bar_u * scale + 1e-30).all(), (np.abs(U - ref) / (scale + 1e-30)).max()
    Y = np.where(U >= 0, 1.0, -1.0) if form % 2 == 0 else U / np.linalg.norm(U, axis=1, keepdims=True)
    ref, scale = (A64.T @ Y.T).T, (abs(A64).T @ np.abs(Y).T).T
    assert (np.abs(V - ref) <= bar_v * scale + 1e-30).all(), (np.abs(V - ref) / (scale + 1e-30)).max()


# few starts (1..8: GEMV; more: 16 x 32 tiles, K split over CTAs or not), the tiles' widths 32, 64, 128, 256
@pytest.mark.parametrize("engine,r", [("simt", r) for r in (1, 2, 5, 8, 9, 16, 17, 33, 70)] +
                         [("tc", r) for r in (1, 31, 32, 33, 64, 65, 128, 129, 256, 257)])
@pytest.mark.parametrize("n,p", [(1, 70), (515, 1027), (1203, 67), (66, 4099)])
def test_product_widths(lib, engine, r, n, p):
    rng = np.random.default_rng(n + 3 * r)
    A = rng.standard_normal((n, p)).astype(np.float32)
    X = rng.standard_normal((r, p)).astype(np.float32)
    h = lib.Handle(A)
    bar = (lambda K: 2e-6) if engine == "simt" else (lambda K: max(2e-6, K / 16.0 * 2.0 ** -23))
    for form in (1, 2):
        U, V = _products(lib, h, form, lib.SPCA_ENGINE_SIMT if engine == "simt" else lib.SPCA_ENGINE_TC, X)
        _check_products(A.astype(np.float64), X, U, V, form, bar(p), bar(n))
    h.close()


def _matrix(n, p, seed):
    if n < 8 or p < 40:
        return np.random.default_rng(seed).standard_normal((n, p)).astype(np.float32)
    return I.spiked_matrix(n, p, I.spiked_thetas(n, p), min(12, p // 8), seed, dtype=np.float32)


def _kw(form, s):
    # (gamma re-targeted in every sweep: a frozen gamma leaves an entry at the threshold, which rounding decides)
    return dict(s=s) if form < 5 else dict(s=s, gamma_target=True, calib=100)


def _solve_matches(lib, oracle, A, form, r, s, sweeps, engine, G=None):
    A64 = A.astype(np.float64)
    p = A.shape[1]
    G = np.random.default_rng(7 * r + p).standard_normal((r, p)).astype(np.float32) if G is None else G
    kw = _kw(form, s)
    h = lib.Handle((A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data, A.shape) if sps.issparse(A) else A)
    out = h.solve(form, r, max_iter=sweeps, tol=-1, x0=G, want_starts=True, engine=engine, **kw)
    h.close()
    ref = oracle.solve(A64, form, G.astype(np.float64), max_iter=sweeps, tol=-1, **kw)
    assert np.array_equal(out["start_status"], ref.status)
    live = ref.status != DEGENERATE
    assert np.array_equal(out["start_iters"][live], ref.iters[live])
    same = (np.abs(out["start_objective"] - ref.f) <= 1e-5 * np.maximum(1.0, np.abs(ref.f))) & \
        (np.abs(out["start_x"] - ref.X).max(axis=1) <= 1e-4)
    assert same[live].sum() >= 0.95 * live.sum(), (same.sum(), r)
    assert abs(out["objective"] - ref.f[ref.best]) <= 1e-5 * max(1.0, abs(ref.f[ref.best]))
    assert np.array_equal(out["support"], np.flatnonzero(out["x"]))
    assert np.array_equal(out["x"], out["start_x"][out["best_start"]])
    return out


# one row per thread while its CTAs are at most 8 per SM (n = 500: 8 CTAs a start), else vectors; rows at
# the edges of a CTA's 64; the y-step inside (n <= 16384) and behind
@pytest.mark.parametrize("n,p,r,form", [(500, 900, 152, 1), (500, 900, 153, 1), (64, 3000, 9, 2), (65, 3000, 9, 5),
                                        (257, 2050, 12, 7), (16384, 70, 9, 3), (16386, 70, 9, 3), (16386, 70, 9, 4)])
def test_gather_shapes(lib, oracle, n, p, r, form):
    _solve_matches(lib, oracle, _matrix(n, p, n + r), form, r, 6, 4, lib.SPCA_ENGINE_TC)


# FP16: two rows per thread while its CTAs are at most 3 per SM (n = 700: 2 CTAs a start), else eight; both
# keep the order of every sum.  (228 and 229 starts share the contractions' tiles and splits, which do depend
# on the number of starts, so the gather alone changes between them.)
def test_gather_shapes_fp16_bits(lib):
    A = _matrix(700, 1500, 5)
    G = np.random.default_rng(3).standard_normal((229, 1500)).astype(np.float32)
    h = lib.Handle(A, storage=lib.SPCA_FP16_RESIDENT)
    few, wide = (h.solve(3, r, s=12, max_iter=6, tol=-1, x0=G[:r], want_starts=True) for r in (228, 229))
    h.close()
    assert np.array_equal(few["start_x"], wide["start_x"][:228])


# CTAs per start fall from 8 to 1 as starts fill the SMs (14 and 15, 33 and 34, 66 and 67, more than one wave)
# and for few columns; columns of A in shared memory or not (500 x 1000, 1000 x 1000); the largest problem
@pytest.mark.parametrize("n,p,r,form", [(100, 500, 14, 1), (100, 500, 15, 2), (37, 301, 33, 3), (37, 301, 34, 4),
                                        (90, 257, 66, 5), (90, 257, 67, 6), (64, 255, 133, 7), (40, 160, 300, 8),
                                        (40, 160, 310, 1), (1, 33, 3, 2), (3, 1, 2, 1), (9, 31, 2, 3), (50, 64, 2, 1),
                                        (500, 1000, 5, 1), (1000, 1000, 9, 3), (1024, 1024, 2, 6), (1024, 1025, 2, 6),
                                        (4, 9000, 3, 1), (9000, 4, 3, 1)])
def test_small_solves(lib, oracle, n, p, r, form):
    _solve_matches(lib, oracle, _matrix(n, p, n + p), form, r, min(p, 8), 3, lib.SPCA_ENGINE_AUTO)


def test_small_solve_degenerate_and_full_pass(lib, oracle):
    A = _matrix(60, 700, 9)
    A[:, 5] = 0.0
    G = np.random.default_rng(1).standard_normal((4, 700)).astype(np.float32)
    G[1] = 0.0
    G[2] = 0.0
    G[2, 5] = 1.0                                            # u = A x = 0
    for form in (1, 3):
        out = _solve_matches(lib, oracle, A, form, 4, 9, 3, lib.SPCA_ENGINE_AUTO, G)
        assert out["degenerate"] == 2
    for form, s in ((1, 650), (3, 640.0)):                   # more survivors than the x-step's list: the full pass
        _solve_matches(lib, oracle, _matrix(60, 1500, 9), form, 4, s, 3, lib.SPCA_ENGINE_AUTO)


# read-backs after 2 sweeps and then every 16 without a tolerance: sweep counts on both sides of each
@pytest.mark.parametrize("sweeps", [1, 2, 3, 18, 19, 35])
@pytest.mark.parametrize("form", [1, 3, 6])
def test_sweep_counts(lib, oracle, sweeps, form):
    A = _matrix(300, 4003, 2)                                # above the one-launch solve
    _solve_matches(lib, oracle, A, form, 40, 12, sweeps, lib.SPCA_ENGINE_TC)


def test_results_copy(lib, oracle):
    """A support past the part that comes with the first copy; x too long for the staged copy; a non-finite
    x0 refused, from host and device memory, and the handle usable after it."""
    import torch
    A = np.random.default_rng(4).standard_normal((300, 4100)).astype(np.float32)
    out = _solve_matches(lib, oracle, A, 1, 2, 3000, 1, lib.SPCA_ENGINE_TC)
    assert out["nnz"] == 3000
    A = np.random.default_rng(5).standard_normal((3, 1 << 20)).astype(np.float32)
    G = np.random.default_rng(6).standard_normal((1, 1 << 20)).astype(np.float32)
    _solve_matches(lib, oracle, A, 1, 1, 20, 1, lib.SPCA_ENGINE_AUTO, G)
    for n, p in ((30, 100), (300, 4100)):
        h = lib.Handle(np.random.default_rng(8).standard_normal((n, p)).astype(np.float32))
        G = np.random.default_rng(9).standard_normal((3, p)).astype(np.float32)
        good = h.solve(1, 3, s=5, max_iter=4, tol=-1, x0=G)
        bad = G.copy()
        bad[1, p - 1] = np.nan
        dev = torch.from_numpy(bad).cuda()
        for kw in (dict(x0=bad), dict(x0=dev.data_ptr(), x0_device=True)):
            with pytest.raises(lib.SpcaError):
                h.solve(1, 3, s=5, max_iter=4, tol=-1, **kw)
            assert np.array_equal(h.solve(1, 3, s=5, max_iter=4, tol=-1, x0=G)["x"], good["x"])
        h.close()


def _rows_of(lengths, p, seed):
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.choice(p, k, replace=False)) for k in lengths]
    ptr = np.concatenate([[0], np.cumsum(lengths)])
    col = np.concatenate(cols) if ptr[-1] else np.zeros(0, int)
    return sps.csr_matrix((rng.integers(1, 9, ptr[-1]).astype(np.float32), col, ptr), shape=(len(lengths), p))


# items of at most 512 entries and 8 rows: rows at those lengths, empty runs, split rows; a lane sums at most
# 16 terms (up to 32 starts; more: an item in order), 5 levels, then the row's segments
@pytest.mark.parametrize("r", [1, 8, 9, 24, 32, 33])
def test_sparse_items(lib, r):
    lengths = [511, 512, 513, 0, 0, 1, 31, 32, 33, 63, 64, 65] + [0] * 20 + [1024, 1025, 5000] + [3] * 50 + [300] * 9
    M = _rows_of(lengths, 6000, r)
    M64 = M.astype(np.float64)
    h = lib.Handle((M.indptr.astype(np.int64), M.indices.astype(np.int32), M.data, M.shape))
    X = np.random.default_rng(r).standard_normal((r, 6000)).astype(np.float32)
    bar = ((16 + 5 if r <= 32 else 512) + 10) * 2.0 ** -24
    for form in (1, 2):
        U, V = _products(lib, h, form, lib.SPCA_ENGINE_AUTO, X)
        _check_products(M64, X, U, V, form, bar, bar)
    h.close()


# the y-step written packed (n > 16384) or not; a support's columns searched by half-warps (at most 32) or
# threads; more starts than a pack tile's 32
@pytest.mark.parametrize("n,r,s", [(16384, 5, 6), (16385, 5, 6), (20001, 33, 32), (20001, 4, 33), (20001, 9, 1)])
def test_sparse_sweeps(lib, oracle, n, r, s):
    rng = np.random.default_rng(n + s)
    M = sps.random(n, 400, density=0.02, format="csr", random_state=rng, dtype=np.float64)
    M.data = rng.integers(1, 9, M.nnz).astype(np.float32)
    M = (sps.csr_matrix(M) + sps.csr_matrix(np.outer(rng.random(n) < 0.05, np.arange(400) < 40) * 3.0)).astype(np.float32).tocsr()
    _solve_matches(lib, oracle, M, 1, r, s, 3, lib.SPCA_ENGINE_AUTO)


# an entry exactly at lambda_s (s = 4.5 and 10, 9, 9, 9, 9 above 8: s sum w^2 = (sum w)^2 at 8) does not survive,
# whether the full pass it is left to runs in the first kernel or in its own
@pytest.mark.parametrize("p", [70, 1025, 8192, 8193, 20011])
@pytest.mark.parametrize("form", [3, 4])
def test_entry_at_lambda(lib, p, form):
    import torch
    rng = np.random.default_rng(p)
    V = np.zeros((3, p), np.float32)
    V[:, 7:] = rng.uniform(-6, 6, (3, p - 7))
    V[:, 1:7] = [10, -9, 9, 8, -9, 9]
    V[2, 4] = 7                                              # the same without the entry
    V = np.roll(V, p // 3, axis=1)
    h = lib.Handle(np.zeros((2, p), np.float32))
    Vd = torch.from_numpy(V).cuda()
    Xd = torch.full((3, p), np.nan, dtype=torch.float32, device="cuda")
    F, T = (torch.zeros(3, dtype=torch.float64, device="cuda") for _ in range(2))
    N = torch.zeros(3, dtype=torch.int32, device="cuda")
    st = lib.spca_xstep(h.h, form, 4.5, 0.0, False, Vd.data_ptr(), p, 3, Xd.data_ptr(), p, F.data_ptr(), N.data_ptr(),
                        T.data_ptr())
    assert st == 0, lib.spca_last_error(h.h)
    h.close()
    w = np.sign(V) * np.maximum(np.abs(V) - 8.0, 0.0)
    assert N.tolist() == [5, 5, 5]
    assert np.abs(Xd.cpu().numpy() - w / np.sqrt(8.0)).max() <= 1e-6
    assert np.abs(T.cpu().numpy() - 8.0).max() <= 1e-6 * 8.0
    assert np.abs(F.cpu().numpy() - (8.0 * np.sqrt(4.5) + np.sqrt(8.0))).max() <= 1e-6 * 20.0
