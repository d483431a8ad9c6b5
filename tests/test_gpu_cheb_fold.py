"""The folded Chebyshev transforms of double-precision plans, nz - 1 a multiple of 8, at the edges of their
register buckets (9, 33 | 41, 65 | 73, 97 | 105, 129 nodes) and beside them (nodes that take the lane
kernels: 34, 37, 99), every wall mode and torque route, boxes whose wavenumbers end inside a block of 16; against
the oracle at the double-precision bar (1e-9)."""

import pytest

from gpu_helpers import gpu_mobility, oracle_params, rel_l2, small_params
from oracle.stokes import mobility
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
