"""F of the x-step is FP64 on the FP32 sum of squares: with one surviving entry w per start, F of T_s and of the
soft threshold is the FP64 square root of fl(w^2), to two units in its last place (2^-51), list and full pass."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,r", [(40, 4096), (3000, 700), (20011, 3)])
@pytest.mark.parametrize("form,full", [(1, False), (7, False), (7, True)])
def test_norm_keeps_fp64(p, r, form, full):
    import torch
    from paper_1212_4137_gb300 import build, spca
    build.build()
    spca.load()
    rng = np.random.default_rng(p + form)
    w = (rng.uniform(1, 2, r) * 2.0 ** rng.integers(-40, 40, r)).astype(np.float32)
    w[:4] = [1.0, 3.0, np.float32(2.0) ** -60, np.float32(2.0) ** 55][:min(4, r)] if r >= 4 else w[:4]
    V = np.zeros((r, p), np.float32)
    V[np.arange(r), rng.integers(0, p, r)] = w
    h = spca.Handle(np.zeros((2, p), np.float32))
    Vd = torch.from_numpy(V).cuda()
    Xd = torch.zeros_like(Vd)
    F, T = (torch.zeros(r, dtype=torch.float64, device="cuda") for _ in range(2))
    N = torch.zeros(r, dtype=torch.int32, device="cuda")
    # (s = p - 1 with the gamma rule: more selected entries than a list takes, so the full pass, gamma = 0)
    s, cal = (float(p - 1), 1) if full else (1.0, 0)
    st = spca.spca_xstep(h.h, form, s, 0.0, cal, Vd.data_ptr(), p, r, Xd.data_ptr(), p, F.data_ptr(), N.data_ptr(),
                         T.data_ptr())
    assert st == 0, spca.spca_last_error(h.h)
    h.close()
    want = np.sqrt((w * w).astype(np.float64))
    assert (np.abs(F.cpu().numpy() - want) <= 2.0 ** -51 * want).all()
    assert (N.cpu().numpy() == 1).all()
