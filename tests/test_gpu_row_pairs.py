"""Row pairs transformed together by one block: ragged last groups (an odd row count, fewer rows than a group
holds, one row left over), rows of one to eight pairs per block and sizes on both sides of each switch, against
the oracle at the parity bars."""

import pytest

from gpu_helpers import gpu_mobility, oracle_params, rel_l2, small_params
from oracle.stokes import mobility
from paper_2210_01837_gb300 import binding
from paper_2210_01837_gb300.workloads import random_particles

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-9, "mixed": 1e-5}


@pytest.mark.parametrize("nx,ny,nz", [
    (12, 12, 9), (32, 15, 33), (48, 35, 17), (64, 49, 13), (96, 27, 17), (128, 25, 13), (160, 45, 9),
    (210, 15, 17), (256, 21, 13), (300, 14, 9), (384, 15, 13), (420, 15, 9), (512, 18, 9), (675, 15, 9),
    (1024, 12, 9), (1280, 15, 9)])
def test_ragged_row_groups_match_oracle(nx, ny, nz):
    params = small_params("bottom_wall", nx=nx, ny=ny, nz=nz, zmax=4.0, torque=True)
    pos, F, T = random_particles(params, 12, seed=nx + ny)
    U_ref, W_ref = mobility(oracle_params(params), pos, F, T)
    for precision in ("fp64", "mixed"):
        plan = binding.Plan.from_params(params, with_torque=True, precision=precision, max_n=len(pos))
        info = plan.info()
        plan.set_fft(0, info.fft_register_cols, info.fft_col_width)
        U, W = gpu_mobility(params, pos, F, T, precision, plan=plan)
        assert rel_l2(U, U_ref) <= TOL[precision], precision
        assert rel_l2(W, W_ref) <= TOL[precision], precision
        plan.close()
