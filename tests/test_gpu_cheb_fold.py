"""The folded Chebyshev transforms of double-precision plans, nz - 1 a multiple of 8, at the edges of their
register buckets (9, 33 | 41, 65 | 73, 97 | 105, 129 nodes) and beside them (nodes that take the lane
kernels: 34, 37, 99), every wall mode and torque route, boxes whose wavenumbers end inside a block of 16; against
the oracle at the double-precision bar (1e-9)."""

import numpy as np
import pytest

from gpu_helpers import gpu_mobility, oracle_params, rel_l2, small_params, to_dev, zrange
from oracle.stokes import mobility
from paper_2210_01837_gb300 import binding
from paper_2210_01837_gb300.workloads import random_particles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("route", [None, "spectral_curl", "kernel_derivative"])
@pytest.mark.parametrize("mode,nx,ny,nz", [
    ("bottom_wall", 16, 14, 9), ("slit", 21, 15, 33), ("free", 16, 12, 33), ("bottom_wall", 15, 14, 34),
    ("slit", 16, 12, 37), ("slit", 16, 12, 41), ("bottom_wall", 18, 14, 65), ("free", 16, 14, 73), ("slit", 15, 12, 97),
    ("bottom_wall", 16, 12, 99), ("free", 16, 12, 105), ("bottom_wall", 16, 12, 129), ("slit", 16, 12, 129)])
def test_folded_transforms_match_oracle(mode, nx, ny, nz, route):
    params = small_params(mode, nx=nx, ny=ny, nz=nz, zmax=4.5, torque=route is not None)
    pos, F, T = random_particles(params, 5, seed=nz, torques=route is not None)
    U_ref, W_ref = mobility(oracle_params(params), pos, F, T, torque_route=route or "spectral_curl")
    U, W = gpu_mobility(params, pos, F, T, "fp64", route=route or "spectral_curl")
    assert rel_l2(U, U_ref) <= 1e-9
    if route is not None:
        assert rel_l2(W, W_ref) <= 1e-9


def sheet(params, n, half, torques):
    """Particles on two planes `half` below and above the middle: the occupied planes are those between."""
    rng = np.random.default_rng(params["nz"])
    pos = rng.uniform(0.0, 1.0, (n, 3)) * [params["Lx"], params["Ly"], 0.0]
    pos[:, 2] = 0.5 * params["zmax"] + half * np.where(np.arange(n) % 2, 1.0, -1.0)
    F, T = rng.standard_normal((2, n, 3))
    return pos, F, T if torques else None


@pytest.mark.parametrize("route", [None, "spectral_curl", "kernel_derivative"])
@pytest.mark.parametrize("mode,nz", [("free", 9), ("slit", 17), ("free", 33), ("free", 65), ("bottom_wall", 73),
                                     ("slit", 97), ("free", 121), ("slit", 121), ("free", 129), ("bottom_wall", 129)])
def test_few_and_many_occupied_planes_match_oracle(mode, nz, route):
    """One plan called with few occupied planes (dense transforms), with some (one direction each way) and with
    most of them (folded), in turn, so that neither kernel leaves the other's planes behind."""
    params = small_params(mode, nx=16, ny=14, nz=nz, zmax=40.0, torque=route is not None)
    kw = dict(with_torque=route or False, precision="fp64", max_n=6)
    plan = binding.Plan.from_params(params, **kw)
    seen = []
    for half in (0.0, 17.0, 3.0, 6.0, 10.0, 0.0):
        pos, F, T = sheet(params, 6, half, route is not None)
        U_ref, W_ref = mobility(oracle_params(params), pos, F, T, torque_route=route or "spectral_curl")
        U, W = gpu_mobility(params, pos, F, T, "fp64", plan=plan)
        lo, hi = zrange(plan)
        seen.append(hi - lo + 1)
        assert rel_l2(U, U_ref) <= 1e-9
        if route is not None:
            assert rel_l2(W, W_ref) <= 1e-9
    plan.close()
    assert min(seen) <= 9 + nz // 10 and max(seen) >= min(nz, 2 * nz // 3)


def test_no_particles_leave_no_flow():
    params = small_params("free", nx=16, ny=14, nz=33, zmax=40.0, torque=False)
    plan = binding.Plan.from_params(params, with_torque=False, precision="fp64", max_n=4)
    plan.apply(*(to_dev(np.zeros((0, 3))) for _ in range(2)), check=True)
    pos, F, _ = sheet(params, 4, 10.0, False)
    U, _ = gpu_mobility(params, pos, F, None, "fp64", plan=plan)
    plan.close()
    U_ref, _ = mobility(oracle_params(params), pos, F, None)
    assert rel_l2(U, U_ref) <= 1e-9


def test_sheet_costs_less_than_a_filled_box():
    """A transform over 3 of 129 planes takes a fraction of the one over all (a fifth here, measured; the
    folded transform alone takes the same time for both)."""
    import torch
    params = small_params("free", nx=256, ny=256, nz=129, zmax=40.0, torque=True)
    plan = binding.Plan.from_params(params, with_torque="spectral_curl", precision="fp64", max_n=100)
    plan.enable_timing(True)
    best = []
    for half in (0.0, 18.0):
        a = [to_dev(x) for x in sheet(params, 100, half, True)]
        t = []
        for _ in range(6):
            plan.apply(*a)
            torch.cuda.synchronize()
            t.append(plan.stage_times()["cheb_fwd"])
        best.append(min(t))
    plan.close()
    assert best[0] < 0.5 * best[1]
