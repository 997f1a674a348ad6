"""Products with A, entry by entry, in every form: rows shared by 1-8 lanes or
sorted within a CTA, one or two columns per thread, columns or rows written,
the allocation-free product. A row has 20 to 175 nonzeros, real coefficients
apart from the boundary's, so a bound taken from the longest row and the
largest entry would let a short row lose its low parts.

Bound of an entry whose row has m nonzeros: its real and imaginary part are
sums of at most 2 m products in any order, each within 2 m u sum |a||x| (u =
2^-53; double-float: 2^-48 with operands split to 2^-47, for which m + 4 <= 2 m
of the same unit), so the complex entry is within 2 sqrt(2) m u sum |a||x|; the
reference adds at most its own FP64 rounding: 4 m u sum |a||x| in all, and
FP64's 6 m 2^-53 where both sides have that unit."""
import numpy as np
import pytest

from paper_2004_07930_gb300 import hz
from paper_2004_07930_gb300 import workloads as wl

from _gpu_common import torch_cuda

pytestmark = pytest.mark.gpu
WIDTHS = (1, 2, 3, 4, 5, 8, 9, 16, 17, 33, 64)


def check(Y, ref, scale, s):
    assert (np.abs(Y - ref[:s]) <= scale[:s]).all(), (s, (np.abs(Y - ref[:s]) / scale[:s]).max())


@pytest.mark.parametrize("precision,unit", [(hz.HZ_PREC_FP64, 6 * 2.0 ** -53), (hz.HZ_PREC_MIXED, 4 * 2.0 ** -48)])
@pytest.mark.parametrize("ncell", [4, 12])  # below and above the size from which a row is one lane's
def test_every_entry_of_a_product(precision, unit, ncell):
    torch = torch_cuda()
    p = wl.cube_problem(ncell=ncell, nparts_xyz=(2, 1, 1), coarse=False)
    with hz.Solver.from_problem(p, coarse_mode=hz.HZ_COARSE_NONE, precision=precision) as S:
        A = S.matrix_csr()
        m = np.diff(A.indptr)
        X = wl.random_rhs(S.n, max(WIDTHS), 62)
        X *= 10.0 ** np.random.default_rng(63).uniform(-3, 3, size=X.shape)   # rows of small and large entries
        ref = (A @ X.T).T
        size = (abs(A) @ np.abs(X).T).T
        scale = unit * m * size
        for s in WIDTHS:
            check(S.apply_A(torch.from_numpy(X[:s]).cuda()).cpu().numpy(), ref, scale, s)
        check(S.apply_A(X[:5]), ref, scale, 5)
        D = torch.from_numpy(X[:3]).cuda()
        if D.numel() <= hz.HZ_NOALLOC_MAX_ENTRIES:
            Y = torch.empty_like(D)
            assert S._lib.hz_apply_A_noalloc(S._ctx, D.data_ptr(), Y.data_ptr(), 3, None) == hz.HZ_OK
            torch.cuda.synchronize()
            check(Y.cpu().numpy(), ref, 6 * 2.0 ** -53 * m * size, 3)   # FP64 in every form
