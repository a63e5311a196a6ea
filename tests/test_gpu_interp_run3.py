"""3D interpolation: the run kernel (eights of coils, and five to seven left over) and the
one-sample-per-thread kernel for the rest, against the float64 oracle: coil counts on both sides of
each rule, sample counts around a warp's batch of 32, its groups of four and the 1024-sample
items, odd k-space strides, many samples in one cell, grids with a ragged last tile and windows
across the periodic edge, every output storage and the dual step."""
import numpy as np
import pytest

from oracle import nufft as onf, solvers as osv
from tests.gpu_util import make_plan, need_gpu, random_problem, rel, rounded, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,C,M,kind", [
    ((16, 16, 16), 8, 1, "c64"), ((16, 12, 20), 5, 31, "bf16"), ((24, 16, 16), 4, 33, "c64"), ((16, 16, 18), 7, 130, "fp16"),
    ((20, 20, 20), 8, 1025, "c64"), ((12, 24, 16), 9, 2051, "c64"), ((16, 16, 16), 13, 700, "bf16"), ((30, 24, 26), 16, 5003, "c64"),
    ((16, 16, 16), 8, 40001, "c64"), ((18, 20, 22), 2, 3001, "c64"), ((16, 16, 16), 1, 9000, "c64"),
])
def test_interpolation_3d(shape, C, M, kind):
    need_gpu()
    x, maps, traj = random_problem(shape, C, M, seed=M, edge=M > 16)
    if M > 64:
        traj[::3] = traj[1]
    m = maps.astype(np.complex128)
    plan = make_plan(shape, C, M)
    plan.set_trajectory(to_dev(traj)).set_maps(to_dev(maps))
    ref = onf.nufft_forward(x.astype(np.complex128), m, traj)
    y = rounded(plan.sense_forward(to_dev(x), storage=kind))
    assert rel(y, ref, "forward") < {"c64": 1e-5, "bf16": 2.0 ** -8, "fp16": 2.0 ** -11}[kind]
    if M < 6000:
        A = lambda v: onf.nufft_forward(v, m, traj)
        AH = lambda v: onf.nufft_adjoint(v, m, traj)
        p = np.full((C, M), 0.5, dtype=np.float32)
        L, _ = osv.power_method(A, AH, p.astype(np.float64), shape, iters=8)
        assert abs(plan.max_eig(to_dev(p), iters=8) / L - 1) < 1e-5
        yc = ref.astype(np.complex64)
        xs = plan.pdhg_solve(to_dev(yc), to_dev(p), "l2", 0.1, 3, lmax=L)[0].cpu().numpy()
        assert rel(xs, osv.pdhg(A, AH, yc, p, shape, "l2", 0.1, 3, L)[0], "dual step") < 1e-5
    plan.close()
