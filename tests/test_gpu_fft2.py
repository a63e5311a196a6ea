"""The own 2D FFT passes with the fused pre-step and combine: forward, adjoint and a few PDHG
iterations against the float64 oracle over the grid lengths they factor differently (one radix
split in two, two to four stages, compiled and summed primes), coil counts that do and do not fill
the lines of a CTA, both line counts per CTA, and every maps storage type."""
import numpy as np
import pytest

from oracle import nufft as onf, solvers as osv
from tests.gpu_util import make_plan, need_gpu, random_problem, rel, rounded, to_dev

pytestmark = pytest.mark.gpu

# (shape, coils, alpha, maps): grids 10x16, 32x256, 300x100, 272x234 (17, 13), 122x62 (61, 31), 140x110 (7, 11),
# 190x78 (19, 13), 500x126, 20x806 (31)
CASES = [((8, 10), 1, 1.25, "c64"), ((16, 128), 2, 2.0, "fp16"), ((240, 80), 3, 1.25, "c64"), ((217, 186), 7, 1.25, "c64"),
         ((97, 49), 30, 1.25, "c64"), ((112, 88), 5, 1.25, "bf16"), ((152, 62), 8, 1.25, "c64"), ((400, 101), 4, 1.25, "c64"),
         ((16, 644), 12, 1.25, "fp16")]


@pytest.mark.parametrize("shape,C,alpha,kind", CASES)
def test_own_2d_fft(shape, C, alpha, kind):
    need_gpu()
    import torch
    from paper_1902_09657_gb300.api import to_storage
    M = 1500
    x, maps, traj = random_problem(shape, C, M, seed=C, edge=True)
    rng = np.random.default_rng(C)
    y = (rng.standard_normal((C, M)) + 1j * rng.standard_normal((C, M))).astype(np.complex64)
    md = to_storage(torch.from_numpy(maps).cuda(), kind)
    m = rounded(md)
    plan = make_plan(shape, C, M, alpha)
    plan.set_trajectory(to_dev(traj)).set_maps(md)
    A = lambda v: onf.nufft_forward(v, m, traj, alpha, 4)
    AH = lambda v: onf.nufft_adjoint(v, m, traj, alpha, 4)
    assert rel(plan.sense_forward(to_dev(x)).cpu().numpy(), A(x.astype(np.complex128)), "forward") < 1e-5
    assert rel(plan.sense_adjoint(to_dev(y)).cpu().numpy(), AH(y.astype(np.complex128)), "adjoint") < 1e-5
    p = np.full((C, M), 0.5, dtype=np.float32)
    L, _ = osv.power_method(A, AH, p.astype(np.float64), shape, iters=30)
    assert abs(plan.max_eig(to_dev(p)) / L - 1) < 1e-5
    for reg, solve in (("l2", osv.pdhg), ("tv", osv.pdhg_tv)):
        ref = (solve(A, AH, y, p, shape, "l2", 0.1, 3, L) if reg == "l2" else solve(A, AH, y, p, shape, 0.1, 3, L))[0]
        xs = plan.pdhg_solve(to_dev(y), to_dev(p), reg, 0.1, 3, lmax=L)[0].cpu().numpy()
        assert rel(xs, ref, reg) < 1e-5
    plan.close()


# grids 26x34x22 (2 13, 2 17, 2 11), 94x38x46 (47, 19, 23), 10x62x90 (31), 60x28x166 (compiled, 7, 83), 14x254x12 (7, 127),
# 48x54x50 (no prime above 5)
@pytest.mark.parametrize("shape,C,kind", [((20, 27, 17), 3, "c64"), ((75, 30, 36), 1, "fp16"), ((8, 49, 72), 8, "c64"),
                                          ((48, 22, 132), 5, "bf16"), ((11, 203, 9), 2, "c64"), ((38, 43, 40), 9, "c64")])
def test_own_3d_fft_of_any_length(shape, C, kind):
    """The 3D passes of run-time length: forward, adjoint and preconditioner (its 2N grids)."""
    need_gpu()
    import torch
    from oracle import precond as opc
    from paper_1902_09657_gb300.api import to_storage
    M = 1200
    x, maps, traj = random_problem(shape, C, M, seed=C, edge=True)
    rng = np.random.default_rng(C)
    y = (rng.standard_normal((C, M)) + 1j * rng.standard_normal((C, M))).astype(np.complex64)
    md = to_storage(torch.from_numpy(maps).cuda(), kind)
    m = rounded(md)
    plan = make_plan(shape, C, M)
    plan.set_trajectory(to_dev(traj)).set_maps(md)
    assert rel(plan.sense_forward(to_dev(x)).cpu().numpy(), onf.nufft_forward(x.astype(np.complex128), m, traj), "forward") < 1e-5
    assert rel(plan.sense_adjoint(to_dev(y)).cpu().numpy(), onf.nufft_adjoint(y.astype(np.complex128), m, traj), "adjoint") < 1e-5
    if C <= 3:
        assert rel(plan.make_preconditioner().cpu().numpy(), opc.mc_precond_fast(m, traj), "preconditioner") < 1e-5
    plan.close()


# 2N grids 20x26 (13), 62x44 (31, 11), 34x96 (17), 48x36; one coil (a lone pair), coil counts that do and do not fill
# the 4 coils of a thread, both line counts per CTA, every maps type
@pytest.mark.parametrize("shape,C,kind", [((10, 13), 1, "c64"), ((31, 22), 3, "fp16"), ((17, 48), 4, "bf16"), ((24, 18), 9, "c64"),
                                          ((64, 50), 13, "c64")])
def test_preconditioner_pairs_and_coils(shape, C, kind):
    """Pair products formed in the row pass, and the denominators of several coils at once."""
    need_gpu()
    import torch
    from oracle import precond as opc
    from paper_1902_09657_gb300.api import to_storage
    M = 700
    _, maps, traj = random_problem(shape, C, M, seed=C, edge=True)
    md = to_storage(torch.from_numpy(maps).cuda(), kind)
    plan = make_plan(shape, C, M)
    plan.set_trajectory(to_dev(traj)).set_maps(md)
    assert rel(plan.make_preconditioner(True).cpu().numpy(), opc.mc_precond_fast(rounded(md), traj), "mc") < 1e-5
    sc = plan.make_preconditioner(False).cpu().numpy()
    ref = opc.sc_precond_fast(traj, shape)
    assert max(rel(sc[c], ref, "sc") for c in range(C)) < 1e-5
    plan.close()
