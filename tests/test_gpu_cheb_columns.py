"""The three-field transforms in registers (mixed precision, no spectral curl): node counts at the edges of
every register bucket and of the two directions' ranges (52 and 68), even and odd, every wall mode, odd grids,
a ragged last block, and a plane range that is not symmetric, against the oracle at the mixed bar."""

import pytest

from gpu_helpers import gpu_mobility, oracle_params, rel_l2, small_params
from oracle.stokes import mobility
from paper_2210_01837_gb300 import binding
from paper_2210_01837_gb300.workloads import random_particles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [8, 9, 19, 20, 21, 35, 36, 37, 51, 52, 53, 67, 68, 69])
@pytest.mark.parametrize("mode,nx,ny", [("bottom_wall", 45, 35), ("slit", 40, 36), ("free", 36, 45)])
def test_register_transforms_match_oracle(mode, nx, ny, nz):
    params = small_params(mode, nx=nx, ny=ny, nz=nz, torque=False)
    pos, F, T = random_particles(params, 20, seed=nx + nz, torques=False)
    U_ref, _ = mobility(oracle_params(params), pos, F, T)
    plan = binding.Plan.from_params(params, with_torque=False, precision="mixed", max_n=len(pos))
    assert plan.info().cheb_tensor_cores == (1 if nz > 52 else 0)
    U, _ = gpu_mobility(params, pos, F, T, "mixed", plan=plan)
    plan.close()
    assert rel_l2(U, U_ref) <= 1e-5


@pytest.mark.parametrize("mode", ["bottom_wall", "slit"])
@pytest.mark.parametrize("nz", [19, 36, 68])
def test_kernel_derivative_route_matches_fp64(mode, nz):
    """Backward in registers, forward on the tensor cores; against the same route in double."""
    params = small_params(mode, nx=45, ny=36, nz=nz, torque=True)
    pos, F, T = random_particles(params, 20, seed=nz)
    out = {}
    for precision in ("mixed", "fp64"):
        plan = binding.Plan.from_params(params, with_torque="kernel_derivative", precision=precision, max_n=len(pos))
        assert plan.info().cheb_tensor_cores == (1 if precision == "mixed" else 0)
        out[precision] = gpu_mobility(params, pos, F, T, precision, plan=plan)
        plan.close()
    assert rel_l2(out["mixed"][0], out["fp64"][0]) <= 1e-5
    assert rel_l2(out["mixed"][1], out["fp64"][1]) <= 1e-5


def test_injected_failure_still_takes_the_tensor_cores():
    """The forward tensor-core transform's failure injection stays available on these plans: the next apply
    takes that transform and reports the expired wait, and the one after it is correct."""
    params = small_params("bottom_wall", nx=40, ny=36, nz=19, torque=False)
    pos, F, T = random_particles(params, 20, seed=3, torques=False)
    U_ref, _ = mobility(oracle_params(params), pos, F, T)
    plan = binding.Plan.from_params(params, with_torque=False, precision="mixed", max_n=len(pos))
    plan.debug_inject(1)
    with pytest.raises(binding.DpsError):
        gpu_mobility(params, pos, F, T, "mixed", plan=plan)
    U, _ = gpu_mobility(params, pos, F, T, "mixed", plan=plan)
    plan.close()
    assert rel_l2(U, U_ref) <= 1e-5
