"""The sum over a long column of a sparse A keeps FP32's last bit: hundreds of segments' sums are added with the
additions' errors, so what is left is each segment's own rounding (a few 2^-24 of a segment, of either sign, over
hundreds of segments) and the final one.  Columns of positive entries and y = +1 (L1 variance, x and A
positive): v is the column's sum, and the root mean square of its relative errors stays below 2^-24, where a
plain sum of the segments comes to 3 times that and more.  Every number of slices that the starts choose."""
import numpy as np
import pytest
import scipy.sparse as sps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [3, 32, 33, 64, 65, 128, 129, 300])
def test_long_column_sums(r):
    import torch
    from paper_1212_4137_gb300 import build, spca
    build.build()
    spca.load()
    n, p, full = 200_000, 40, 24
    rng = np.random.default_rng(r)
    A = np.zeros((n, p), np.float32)
    A[:, :full] = rng.uniform(1, 2, (n, full))
    A[:700, full] = 1.5                                      # two segments, and short columns
    A[3, full + 1:] = 2.0
    M = sps.csr_matrix(A)
    h = spca.Handle((M.indptr.astype(np.int64), M.indices.astype(np.int32), M.data, M.shape))
    X = torch.rand(r, p, device="cuda") + 0.1
    U, V = torch.zeros(r, n, device="cuda"), torch.zeros(r, p, device="cuda")
    st = spca.spca_products(h.h, 2, spca.SPCA_ENGINE_AUTO, X.data_ptr(), p, r, U.data_ptr(), n, V.data_ptr(), p)
    assert st == 0, spca.spca_last_error(h.h)
    h.close()
    want = A.astype(np.float64).sum(axis=0)
    rel = V.cpu().numpy() / want - 1.0
    assert np.sqrt((rel[:, :full] ** 2).mean()) <= 2.0 ** -24, np.sqrt((rel[:, :full] ** 2).mean())
    assert np.abs(rel).max() <= 4 * 2.0 ** -24
    assert (rel == rel[0]).all()                             # the same sums for every start
