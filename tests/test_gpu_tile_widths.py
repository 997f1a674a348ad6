"""Widths of the tile form of the front sweeps (tensor_cores = 1, blocks of 9-16
columns, rows of the block's own width): every column of a narrower block has
the bits of the same column in a block of 16, in either order of the calls."""
import numpy as np
import pytest

from paper_2004_07930_gb300 import hz
from paper_2004_07930_gb300 import workloads as wl

from _gpu_common import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coarse", [hz.HZ_COARSE_NONE, hz.HZ_COARSE_GMRES])
def test_tile_form_at_every_width(coarse):
    torch_cuda()
    p = wl.cube_problem(ncell=6, nparts_xyz=(2, 2, 1))
    with hz.Solver.from_problem(p, precision=hz.HZ_PREC_MIXED, coarse_mode=coarse, tensor_cores=1) as S:
        X = wl.random_rhs(S.n, 16, 61)
        first = S.apply_prec(X[:9])
        ref = S.apply_prec(X)
        np.testing.assert_array_equal(first, ref[:9])
        for s in (9, 11, 12, 13, 15):
            np.testing.assert_array_equal(S.apply_prec(X[:s]), ref[:s])
