"""A member of a group gives the same bits alone and in any mix, also where the mix changes the CTA size
of the grouped x-step (the group's starts and its longest v choose it) and the member's results do not fit
the x-step's list with room to spare: T_s with s near 500, lambda_s with s = 140, gamma targeting, short v."""
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


# (n, p, form, s, r, storage of a resident 16-bit handle)
MEMBERS = [(300, 5000, 1, 500, 48, False), (300, 5000, 3, 140, 48, False), (200, 2500, 4, 60, 40, False),
           (150, 600, 3, 20, 33, False), (150, 900, 2, 350, 40, False), (250, 7000, 7, 480, 48, False),
           (120, 1021, 3, 100, 17, False), (300, 5000, 3, 140, 20, True), (250, 9000, 6, 470, 30, False)]


def _same(a, b, what):
    for k in ("start_x", "start_F", "start_gamma", "start_iters", "start_status", "start_objective",
              "start_explained", "x", "y", "support"):
        assert np.array_equal(a[k], b[k]), (what, k)
    assert a["best_start"] == b["best_start"] and a["objective"] == b["objective"], what


@pytest.mark.parametrize("companion", ["many_starts", "long_v"])
def test_group_member_bits_do_not_depend_on_the_mix(lib, companion):
    handles, reqs = [], []
    for i, (n, p, form, s, r, h16) in enumerate(MEMBERS):
        A = I.spiked_matrix(n, p, I.spiked_thetas(n, p, (40.0, 30.0, 20.0)), 20, 7100 + i, dtype=np.float32)
        h = lib.Handle(A, storage=lib.SPCA_FP16_RESIDENT if h16 else lib.SPCA_F32)
        kw = dict(s=float(s), seed=40 + i, max_iter=7, tol=-1)
        if form >= 5:
            kw.update(gamma_target=True, calib=4)
        handles.append(h)
        reqs.append((h, form, r, kw))
    if companion == "many_starts":       # past three starts per SM: the smallest CTAs
        n, p, r = 100, 800, 600
    else:                                # v beyond 131072 entries: the largest CTAs, while starts are few
        n, p, r = 40, 140001, 3
    A = np.random.default_rng(5).standard_normal((n, p)).astype(np.float32)
    other = lib.Handle(A)
    handles.append(other)
    extra = (other, 1, r, dict(s=12.0, seed=9, max_iter=7, tol=-1))
    g = lib.Group()
    for i, q in enumerate(reqs):
        alone = g.solve([q], want_starts=True)[0]
        mixed = g.solve([q, extra], want_starts=True)[0]
        _same(alone, mixed, (companion, MEMBERS[i]))
    together = g.solve(reqs + [extra], want_starts=True)
    alone = [g.solve([q], want_starts=True)[0] for q in reqs]
    for i, (a, t) in enumerate(zip(alone, together)):
        _same(a, t, (companion, "all", MEMBERS[i]))
    g.close()
    for h in handles:
        h.close()
