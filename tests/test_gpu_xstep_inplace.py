"""spca_xstep with X = V: each row is read before its result replaces it, so the call gives the bits that
it gives into another buffer.  Results from the short list and from the full pass, v in shared memory and
beyond it, rows of every alignment, few and many starts."""
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


def _xstep(lib, h, form, s, cal, gamma, V, X, r):
    import torch
    F, T = (torch.zeros(r, dtype=torch.float64, device="cuda") for _ in range(2))
    N = torch.zeros(r, dtype=torch.int32, device="cuda")
    st = lib.spca_xstep(h.h, form, float(s), gamma, cal, V.data_ptr(), V.stride(0), r, X.data_ptr(), X.stride(0),
                        F.data_ptr(), N.data_ptr(), T.data_ptr())
    assert st == 0, lib.spca_last_error(h.h)
    return F, N, T


@pytest.mark.parametrize("p,ld,r", [(50, 50, 3), (701, 703, 5), (3001, 3001, 480), (8192, 8196, 4), (20011, 20013, 7),
                                    (20011, 20011, 500), (60001, 60001, 3)])
def test_xstep_in_place(lib, p, ld, r):
    import torch
    g = torch.Generator(device="cuda").manual_seed(p + r)
    V = torch.randn(r, ld, generator=g, device="cuda") * 3
    V[:, 5::97] *= 3
    V[0, :p] = 0
    V[1, ::3] = 0
    h = lib.Handle(np.zeros((2, p), np.float32))
    for form in range(1, 9):
        for s in sorted({1, min(p, 40), min(p, 300), min(p, 900), p}):
            for cal in ((0, 1) if form >= 5 else (0,)):
                gamma = 4.0 if form >= 5 and not cal else 0.0
                X = torch.full((r, ld), float("nan"), device="cuda")
                a = _xstep(lib, h, form, s, cal, gamma, V, X, r)
                W = V.clone()
                b = _xstep(lib, h, form, s, cal, gamma, W, W, r)
                assert torch.equal(X[:, :p], W[:, :p]), (form, s, cal)
                assert torch.equal(V[:, p:], W[:, p:])
                for t, u in zip(a, b):
                    assert torch.equal(t, u), (form, s, cal)
    h.close()
