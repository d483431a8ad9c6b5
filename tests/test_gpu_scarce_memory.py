"""Plan creation with too little device memory for the tables that a plan can run without: they are left out,
in the order folded transforms, solve, and the product is that of the plan that has them, to the parity bars
(1e-9 in double, 1e-5 in mixed precision).  A block of memory held by the test leaves the plan what it needs
and half of the last table that does not fit (30 to 130 MB)."""

import gc

import pytest

from gpu_helpers import gpu_mobility, rel_l2, small_params
from paper_2210_01837_gb300 import binding
from paper_2210_01837_gb300.workloads import random_particles

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-9, "mixed": 1e-5}


def tables(nx, ny, nz, precision, tiled):
    """Bytes of the optional tables of a no-slip plan in the order in which they are given up."""
    kp = (nx // 2 + 1) * (ny // 2 + 1)
    size = 8 if precision == "fp64" else 4
    solve = kp * (nz * (32 + size) + 112) if tiled else kp * nz * 32
    return [kp * nz * 16, solve] if precision == "fp64" and (nz - 1) % 8 == 0 else [solve]


@pytest.mark.parametrize("nx,ny,nz,precision,tiled,without", [
    (512, 512, 97, "mixed", False, 1), (384, 384, 97, "fp64", False, 1), (384, 384, 97, "fp64", False, 2),
    (1024, 1024, 49, "mixed", True, 1)])
def test_tables_give_way_to_what_the_plan_needs(nx, ny, nz, precision, tiled, without):
    import torch
    params = small_params("slit", nx=nx, ny=ny, nz=nz, zmax=10.0, torque=False)
    pos, F, _ = random_particles(params, 50, seed=nz, torques=False)
    kw = dict(with_torque=False, precision=precision, max_n=len(pos))
    plan = binding.Plan.from_params(params, **kw)
    full = plan.info().device_bytes
    U_ref, _ = gpu_mobility(params, pos, F, None, precision, plan=plan)
    plan.close()
    lost = tables(nx, ny, nz, precision, tiled)[:without]
    # a tiled plan without its table takes the other solves' workspace, 456 blocks of 128 wavenumbers
    instead = 456 * 128 * nz * (3 * 16 + 3 * 8 + 8) if tiled else 0
    needs = full - sum(lost) + instead
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = needs + (lost[-1] - instead) // 2
    held = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        plan = binding.Plan.from_params(params, **kw)
        small = plan.info().device_bytes
        U, _ = gpu_mobility(params, pos, F, None, precision, plan=plan)
        plan.close()
    finally:
        del held
        torch.cuda.empty_cache()
    assert abs(small - needs) < 1 << 20
    assert rel_l2(U, U_ref) <= TOL[precision]
