"""u = A x over the union of the supports (many rows of A, starts that share few columns), in tiles of every
width: after the first read-back the launches of the union are made in every sweep, and it is taken because
the supports lie in fewer columns than it holds.  Solves of 7 sweeps against FP64 (plain torch), with the bars
of test_gpu_paths: at least 95 % of the starts with the objective within 1e-5 and x within 1e-4, the best
objective within 1e-5."""
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


def _reference(A, X0, s, sweeps):
    A = A.double()
    X = X0.double() / X0.double().norm(dim=1, keepdim=True)
    for _ in range(sweeps):
        U = X @ A.T
        V = (U / U.norm(dim=1, keepdim=True)) @ A
        at = V.abs().topk(s, dim=1).indices
        W = V.new_zeros(V.shape).scatter_(1, at, V.gather(1, at))
        X = W / W.norm(dim=1, keepdim=True)
    return X.cpu().numpy(), (X @ A.T).norm(dim=1).cpu().numpy()


# (n, p, starts, s, strong columns): n times the sum of the supports above 2^29, that sum at most 2^14, s at most
# p / 16 (else the dense u = A x is queued); tiles of 32, 64, 128 and 256 columns
@pytest.mark.parametrize("n,p,r,s,strong", [(67200, 4000, 32, 250, 400), (97000, 1400, 64, 87, 150),
                                            (48403, 1400, 128, 87, 150), (33001, 1403, 188, 87, 150)])
@pytest.mark.parametrize("form", [1, 5])
def test_union_of_supports(lib, n, p, r, s, strong, form):
    import torch
    sweeps = 7
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn(n, p, generator=g, device="cuda")
    cols = torch.randperm(p, generator=g, device="cuda")[:strong]
    A[:, cols] *= 3 + 2 * torch.rand(strong, generator=g, device="cuda")
    X0 = torch.randn(r, p, generator=g, device="cuda")
    h = lib.Handle(A)
    before = h.profile_query(lib.SPCA_K_U_SPARSE)[0]
    kw = dict(gamma_target=True, calib=sweeps) if form == 5 else {}
    out = h.solve(form, r, s=float(s), max_iter=sweeps, tol=-1, x0=X0.data_ptr(), x0_device=True,
                  engine=lib.SPCA_ENGINE_TC, want_starts=True, **kw)
    # a gather per sweep; from the third on the marks and their scan (2), from the fourth on the contraction (3)
    assert h.profile_query(lib.SPCA_K_U_SPARSE)[0] - before == sweeps + 2 * (sweeps - 2) + 3 * (sweeps - 3)
    h.close()
    assert np.count_nonzero((out["start_x"] != 0).any(axis=0)) <= min(1024, (p + 63) // 64 * 64)
    assert n * int((out["start_x"] != 0).sum()) >= 2 ** 29
    X, norm = _reference(A, X0, s, sweeps)
    f = out["start_explained"] if form == 5 else out["start_objective"]
    want = norm ** 2 if form == 5 else norm
    same = (np.abs(f - want) <= 1e-5 * want) & (np.abs(out["start_x"] - X).max(axis=1) <= 1e-4)
    assert same.mean() >= 0.95, same.mean()
    assert abs(out["explained_variance"] - (norm ** 2).max()) <= 2e-5 * (norm ** 2).max()
