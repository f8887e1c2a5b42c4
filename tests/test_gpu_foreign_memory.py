"""Device arguments outside this GPU's own memory (x0 of a solve, X, U and V of spca_products) go by a copy, as
another GPU's memory has to, which kernels cannot use without peer access; here page-locked host memory
stands for it.  The results have the bits of device memory's."""
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


@pytest.mark.parametrize("n,p,r", [(60, 301, 5), (700, 4099, 40)])
def test_x0_elsewhere(lib, n, p, r):
    import torch
    rng = np.random.default_rng(p)
    h = lib.Handle(rng.standard_normal((n, p)).astype(np.float32))
    x0 = torch.from_numpy(rng.standard_normal((r, p)).astype(np.float32))
    kw = dict(s=9.0, max_iter=5, tol=-1, x0_device=True, want_starts=True)
    here, there = x0.cuda(), x0.pin_memory()
    a, b = (h.solve(3, r, x0=t.data_ptr(), **kw) for t in (here, there))
    assert np.array_equal(a["start_x"], b["start_x"]) and a["objective"] == b["objective"]
    there[1, 2] = float("nan")
    with pytest.raises(lib.SpcaError) as e:
        h.solve(3, r, x0=there.data_ptr(), **kw)
    assert e.value.status == lib.SPCA_E_INVALID
    h.close()


def test_products_elsewhere(lib):
    import torch
    n, p, r = 301, 2050, 33
    rng = np.random.default_rng(1)
    h = lib.Handle(rng.standard_normal((n, p)).astype(np.float32))
    X = torch.from_numpy(rng.standard_normal((r, p + 3)).astype(np.float32))
    out = []
    for move in (lambda t: t.cuda(), lambda t: t.pin_memory()):
        x, u, v = move(X), move(torch.zeros(r, n + 5)), move(torch.zeros(r, p + 1))
        st = lib.spca_products(h.h, 1, lib.SPCA_ENGINE_AUTO, x.data_ptr(), p + 3, r, u.data_ptr(), n + 5, v.data_ptr(),
                               p + 1)
        assert st == 0, lib.spca_last_error(h.h)
        torch.cuda.synchronize()
        out.append((u.cpu(), v.cpu()))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert out[0][0][:, :n].abs().sum() > 0 and (out[0][0][:, n:] == 0).all()
    h.close()
