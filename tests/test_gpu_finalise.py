"""The objectives of a solve at the sizes where the finalise changes: the rows of a chunk (one or four per
thread) by the problem's rows and starts, edges of the chunks, FP32 and 16-bit A, supports of a few columns
and of all of them.  A holds whole numbers, which the 16-bit copy keeps, so every objective is compared with
the FP64 one of the returned x; u is summed in compensated FP32 pairs (2^-44 relative to sum |a x| per entry),
so 1e-11 of the objective's size is far above its error and far below FP32's."""
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


@pytest.mark.parametrize("n,r", [(1, 3), (127, 2), (128, 700), (129, 5), (256, 608), (257, 607), (257, 608), (511, 610),
                                 (512, 607), (512, 609), (513, 303), (513, 304), (513, 305), (2100, 121), (2100, 122)])
@pytest.mark.parametrize("resident", [False, True])
def test_objectives_at_chunk_edges(lib, n, r, resident):
    p = 300
    rng = np.random.default_rng(n + r)
    A = rng.integers(-8, 9, (n, p)).astype(np.float32)
    A64 = A.astype(np.float64)
    h = lib.Handle(A, storage=lib.SPCA_FP16_RESIDENT if resident else lib.SPCA_F32)
    for form, s in ((1, 9), (2, 300), (7, 150)):
        kw = dict(gamma_target=True, calib=5) if form == 7 else {}
        out = h.solve(form, r, s=float(s), max_iter=2, tol=-1, seed=3, want_starts=True, **kw)
        X = out["start_x"].astype(np.float64)
        U = X @ A64.T
        norm = np.abs(U).sum(1) if form == 2 else np.linalg.norm(U, axis=1)
        f = norm - (out["start_gamma"] * np.abs(X).sum(1) if form == 7 else 0.0)
        ev = norm if form == 2 else norm ** 2
        scale = np.maximum(norm, 1.0)
        assert (np.abs(out["start_objective"] - f) <= 1e-11 * scale).all()
        assert (np.abs(out["start_explained"] - ev) <= 1e-11 * np.maximum(ev, 1.0)).all()
        best = out["best_start"]
        assert best == int(np.argmax(out["start_explained"] if form == 7 else out["start_objective"]))
    h.close()


def test_group_objectives_alone_and_in_a_mix(lib):
    rng = np.random.default_rng(4)
    sizes = [(257, 400, 500), (2100, 300, 122), (100, 500, 40), (600, 300, 300)]
    handles = [lib.Handle(rng.integers(-8, 9, (n, p)).astype(np.float32)) for n, p, _ in sizes]
    reqs = [(h, 1 + i % 2, r, dict(s=7.0 + 40 * i, seed=i, max_iter=2 + i, tol=-1))
            for i, (h, (_, _, r)) in enumerate(zip(handles, sizes))]
    g = lib.Group()
    alone = [g.solve([q], want_starts=True)[0] for q in reqs]
    for a, t in zip(alone, g.solve(reqs, want_starts=True)):
        assert np.array_equal(a["start_objective"], t["start_objective"])
        assert np.array_equal(a["start_explained"], t["start_explained"]) and a["best_start"] == t["best_start"]
        assert np.array_equal(a["y"], t["y"]) and np.array_equal(a["x"], t["x"])
    g.close()
    for h in handles:
        h.close()
