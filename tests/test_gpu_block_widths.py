"""Block widths, leaf sizes and restart lengths at the edges of the kernels'
splits: the front sweeps work on column blocks of 1, 2, 4, 8 and 16 and on
groups of 16 front rows, the products give a row to 1-8 lanes or a thread two
columns, the Gram-Schmidt products take 12 vectors per launch. Every case against the
oracle's operators: local solves within 1e-9 (FP64) and 1e-5 (FP32) relative
L2 and wavefields within 1e-8 at rtol 1e-10, the bounds of the parity tests;
a product's row of m terms within 2 m eps sum |a x|, eps = 2^-53 (FP64) or
2^-48 (double-float)."""
import numpy as np
import pytest

from oracle import assemble as oa
from oracle import schwarz as osw
from paper_2004_07930_gb300 import hz
from paper_2004_07930_gb300 import workloads as wl

from _gpu_common import dof_perm, rel_l2, torch_cuda

pytestmark = pytest.mark.gpu
WIDTHS = (1, 2, 3, 4, 5, 8, 9, 16, 17, 24, 33, 48, 64)


@pytest.fixture(scope="module")
def cube():
    torch_cuda()
    p = wl.cube_problem(ncell=4, nparts_xyz=(2, 1, 1), top_dirichlet=True)
    return p, osw.TwoLevel(p, coarse_mode="none")


@pytest.mark.parametrize("precision", [hz.HZ_PREC_FP64, hz.HZ_PREC_MIXED])
@pytest.mark.parametrize("leaf", [3, 40, 64, 5000])  # 5000: one front per subdomain (k = f > 128)
def test_local_solves_at_every_width(cube, precision, leaf):
    p, T = cube
    bound = 1e-9 if precision == hz.HZ_PREC_FP64 else 1e-5
    with hz.Solver.from_problem(p, coarse_mode=hz.HZ_COARSE_NONE, precision=precision, leaf_size=leaf,
                                debug_bounds=1) as S:
        perm = dof_perm(S, T.space, 1000.0)
        back = np.argsort(perm)
        X = wl.random_rhs(S.n, max(WIDTHS), 31)
        ref = T.apply(X[:, back].T).T[:, perm]
        for s in WIDTHS:
            Y = S.apply_prec(X[:s])
            assert rel_l2(Y, ref[:s]).max() <= bound, s


@pytest.mark.parametrize("precision", [hz.HZ_PREC_FP64, hz.HZ_PREC_MIXED])
@pytest.mark.parametrize("ncell", [4, 12])  # below and above the size from which a row is one lane's
def test_products_at_every_width(precision, ncell):
    torch = torch_cuda()
    p = wl.cube_problem(ncell=ncell, nparts_xyz=(2, 1, 1), coarse=False)
    with hz.Solver.from_problem(p, coarse_mode=hz.HZ_COARSE_NONE, precision=precision) as S:
        A = S.matrix_csr()
        X = wl.random_rhs(S.n, max(WIDTHS), 32)
        ref = (A @ X.T).T
        eps = 2.0 ** (-53 if precision == hz.HZ_PREC_FP64 else -48)
        bound = 2 * np.diff(A.indptr).max() * eps * (abs(A) @ np.abs(X.T)).max()
        for s in WIDTHS:
            for Y in (S.apply_A(X[:s]), S.apply_A(torch.from_numpy(X[:s]).cuda()).cpu().numpy()):
                assert np.abs(Y - ref[:s]).max() <= bound, s
        # in place: input and output are one buffer
        for s in (1, 5):
            D = torch.from_numpy(X[:s].copy()).cuda()
            assert S._lib.hz_apply_A(S._ctx, D.data_ptr(), D.data_ptr(), s, 1) == hz.HZ_OK
            assert np.abs(D.cpu().numpy() - ref[:s]).max() <= bound, s


def test_allocation_free_product_of_many_columns():
    torch = torch_cuda()
    p = wl.cube_problem(ncell=2, nparts_xyz=(1, 1, 1), coarse=False)
    with hz.Solver.from_problem(p, coarse_mode=hz.HZ_COARSE_NONE) as S:
        A = S.matrix_csr()
        for s in (65, 300, 1100):
            X = wl.random_rhs(S.n, s, 33)
            D = torch.from_numpy(X).cuda()
            Y = torch.empty_like(D)
            assert S._lib.hz_apply_A_noalloc(S._ctx, D.data_ptr(), Y.data_ptr(), s, None) == hz.HZ_OK
            torch.cuda.synchronize()
            ref = (A @ X.T).T
            bound = 2 * np.diff(A.indptr).max() * 2.0 ** -53 * (abs(A) @ np.abs(X.T)).max()
            assert np.abs(Y.cpu().numpy() - ref).max() <= bound, s


@pytest.mark.parametrize("precision,emulate", [(hz.HZ_PREC_FP64, 1), (hz.HZ_PREC_MIXED, 1), (hz.HZ_PREC_MIXED, 0)])
@pytest.mark.parametrize("restart,parts", [(7, (2, 1, 1)), (40, (4, 4, 4)), (1500, (4, 4, 4))])
def test_restart_lengths(cube, precision, emulate, restart, parts):
    """Several cycles; more than one launch of basis vectors; per-column
    scratch beyond shared memory."""
    p, _ = cube
    rng = np.random.default_rng(34)
    src = rng.uniform(150.0, 850.0, size=(3, 3))
    space, A, F = oa.system(p["fine"], p["velocity"], p["freq"], src)
    u_or = oa.solve(A, F)
    # many small subdomains: a preconditioner weak enough for more than 32 steps
    q = wl.cube_problem(ncell=4, nparts_xyz=parts, top_dirichlet=True, coarse=False)
    with hz.Solver.from_problem(q, coarse_mode=hz.HZ_COARSE_NONE, precision=precision, emulate_fp64=emulate,
                                restart=restart, rtol=1e-10, maxit=2000) as S:
        perm = dof_perm(S, space, 1000.0)
        u, st = S.solve(src)
        print("restart", restart, "iterations", st["iterations"])
        assert st["converged"] == 1
        assert rel_l2(u, u_or[:, perm]).max() <= 1e-8
