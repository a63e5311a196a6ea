"""Run spreading (variants 13 and 14): the adjoint against the float64 oracle at the sizes where it can go
wrong: sample counts around the 32-sample staging rounds and the runs of one warp and one CTA, coil
groups of 8 and the narrow lane layouts of the last group, grid widths that are and are not
multiples of the four-column blocks, windows across the periodic edge, many samples in one cell,
and every storage type of the samples."""
import numpy as np
import pytest

from tests.gpu_util import make_plan, need_gpu, random_problem, rel, rounded, to_dev
from oracle import nufft as onf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,C,M,kind", [
    ((16, 16), 1, 1, "c64"), ((16, 18), 2, 31, "c64"), ((21, 34), 3, 32, "bf16"), ((40, 24), 4, 33, "c64"),
    ((33, 33), 5, 255, "fp16"), ((64, 50), 8, 257, "c64"), ((48, 75), 9, 2049, "c64"), ((24, 24), 12, 5000, "bf16"),
    ((96, 96), 32, 3001, "c64"), ((12, 12), 6, 160000, "c64"),
])
def test_run_spreading_matches_oracle(shape, C, M, kind, monkeypatch):
    need_gpu()
    import torch
    from paper_1902_09657_gb300.api import to_storage
    monkeypatch.setenv("KPDHG_SPREAD_VARIANT", "13")
    monkeypatch.setenv("KPDHG_SPREAD_CHUNK", "256")
    _, maps, traj = random_problem(shape, C, M, seed=M + C, edge=M > 16)
    if M > 64:
        traj[:: 3] = traj[0]                       # a third of the samples share one cell
    rng = np.random.default_rng(M)
    y = (rng.standard_normal((C, M)) + 1j * rng.standard_normal((C, M))).astype(np.complex64)
    plan = make_plan(shape, C, M)
    plan.set_trajectory(to_dev(traj)).set_maps(to_dev(maps))
    assert plan.spread_config()["variant"] == 13
    yd = to_storage(torch.from_numpy(y).cuda(), kind)
    ref = onf.nufft_adjoint(rounded(yd), maps.astype(np.complex128), traj)
    for _ in range(2):                             # the second call starts from a used grid
        assert rel(plan.sense_adjoint(yd).cpu().numpy(), ref, "run spreading") < 1e-5
    plan.close()


@pytest.mark.parametrize("shape,C,M,kind", [
    ((16, 16, 16), 8, 1, "c64"), ((20, 16, 20), 5, 63, "bf16"), ((16, 20, 20), 1, 64, "c64"), ((24, 16, 18), 2, 65, "fp16"),
    ((20, 20, 20), 4, 129, "c64"), ((12, 24, 16), 9, 2051, "c64"), ((16, 16, 16), 11, 700, "bf16"), ((30, 24, 26), 16, 5003, "c64"),
    ((8, 9, 10), 6, 3000, "c64"), ((16, 16, 16), 8, 40001, "c64"),
])
def test_run_spreading_3d_matches_oracle(shape, C, M, kind):
    need_gpu()
    import torch
    from paper_1902_09657_gb300.api import to_storage
    _, maps, traj = random_problem(shape, C, M, seed=M + C, edge=M > 16)
    if M > 64:
        traj[::3] = traj[0]
    rng = np.random.default_rng(M)
    y = (rng.standard_normal((C, M)) + 1j * rng.standard_normal((C, M))).astype(np.complex64)
    plan = make_plan(shape, C, M)
    plan.set_trajectory(to_dev(traj)).set_maps(to_dev(maps))
    assert plan.spread_config()["variant"] == 14
    yd = to_storage(torch.from_numpy(y).cuda(), kind)
    ref = onf.nufft_adjoint(rounded(yd), maps.astype(np.complex128), traj)
    for _ in range(2):
        assert rel(plan.sense_adjoint(yd).cpu().numpy(), ref, "run spreading 3D") < 1e-5
    plan.close()
