"""One column through the front sweeps. A column's arithmetic does not depend
on the block it is in, so a block of one column, which has kernels of its own
(FP64: the real and the imaginary part on two lanes; FP32: long reductions of
few fronts cut by chunks of 128 over a CTA's warps), gives the bits of the same
column in a block of two. Sizes: one front per subdomain of 343, 1000 and 2197
rows (3, 8 and 18 chunks, whole and cut by the groups of 16), and trees with
short and long fronts."""
import numpy as np
import pytest

from paper_2004_07930_gb300 import hz
from paper_2004_07930_gb300 import workloads as wl

from _gpu_common import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [hz.HZ_PREC_FP64, hz.HZ_PREC_MIXED])
@pytest.mark.parametrize("ncell,parts,leaf", [(2, (1, 1, 1), 5000), (3, (1, 1, 1), 5000), (4, (1, 1, 1), 5000),
                                              (4, (2, 1, 1), 300), (6, (2, 2, 1), 64), (6, (1, 1, 1), 200)])
def test_one_column_equals_the_column_of_a_block(precision, ncell, parts, leaf):
    torch_cuda()
    p = wl.cube_problem(ncell=ncell, nparts_xyz=parts, coarse=False)
    with hz.Solver.from_problem(p, coarse_mode=hz.HZ_COARSE_NONE, precision=precision, leaf_size=leaf) as S:
        X = wl.random_rhs(S.n, 2, 60)
        Y1, Y2 = S.apply_prec(X[:1]), S.apply_prec(X)
        assert np.isfinite(Y1).all()
        np.testing.assert_array_equal(Y1[0], Y2[0])
