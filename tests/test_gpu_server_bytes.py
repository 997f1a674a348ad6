"""hz_server_column_bytes: a server of whole column blocks (1, 2, 4, 8, 16 or a
multiple of 8 slots) holds no more device memory than its slots times that
figure and the staging column, and a server of any other number no more than
one of the next such number (its sub-vectors and front vectors have that many
columns: 16 at 9 slots). `device_bytes` counts the context; the server's B, X
and R blocks and its staging column, complex128 of n rows each, come on top."""
import pytest

from paper_2004_07930_gb300 import hz
from paper_2004_07930_gb300 import workloads as wl

from _gpu_common import torch_cuda

pytestmark = pytest.mark.gpu
M, D = hz.HZ_PREC_MIXED, hz.HZ_PREC_FP64
N, G, E = hz.HZ_COARSE_NONE, hz.HZ_COARSE_GMRES, hz.HZ_COARSE_DIRECT
WHOLE = (1, 2, 4, 8, 16, 24, 32, 40, 48, 56, 64)


@pytest.mark.parametrize("opts", [
    dict(precision=D, coarse_mode=N, restart=3), dict(precision=M, coarse_mode=N, restart=3),
    dict(precision=D, coarse_mode=G), dict(precision=M, coarse_mode=G), dict(precision=M, coarse_mode=E),
    dict(precision=M, coarse_mode=G, coarse_fp32=1), dict(precision=M, coarse_mode=G, emulate_fp64=0),
    dict(precision=M, coarse_mode=N, tensor_cores=1), dict(precision=M, coarse_mode=N, recycle=8),
    dict(precision=D, coarse_mode=N, block_arnoldi=1, max_block=32)],
    ids=lambda o: "-".join(str(v) for v in o.values()))
def test_servers_stay_within_their_slots_bytes(opts):
    torch_cuda()
    p = wl.cube_problem(ncell=4)
    with hz.Solver.from_problem(p, **opts) as S:
        base = S.info()["device_bytes"]
        for slots in (1, 2, 3, 5, 8, 9, 16, 17, 25, 33, 64):   # the workspace grows from one to the next
            if slots > S.options.max_block:
                continue
            srv = hz.Server(S, slots)
            held = S.info()["device_bytes"] - base + 16.0 * S.n * 3 * slots   # without the staging column
            srv.close()
            whole = next(w for w in WHOLE if w >= slots)
            print(slots, held / whole / S.column_bytes())
            assert held <= whole * S.column_bytes(), slots
            if whole == slots and not (S.options.block_arnoldi or S.options.recycle):   # exact, to the MB
                assert held >= slots * S.column_bytes() - 2.0 ** 20, slots
