"""The tiled solve at the edges of its ranges: fewest and most nodes, even and odd node counts (parities
of unequal length, rows short of whole batches), boxes whose wavenumbers end inside a tile or fill fewer
tiles than a block, odd sizes without Nyquist columns, and the first node count past it; each against
the oracle at the parity bars (1e-9 in double, 1e-5 in mixed precision)."""

import pytest

from oracle.stokes import mobility
from paper_2210_01837_gb300.workloads import random_particles
from gpu_helpers import gpu_mobility, oracle_params, rel_l2, small_params

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-9, "mixed": 1e-5}

# nx, ny, nz, zmax: the spacing is fixed, so short columns take low boxes
SHAPES = [(16, 12, 7, 4.0), (21, 15, 8, 4.0), (20, 14, 26, 6.0), (27, 25, 34, 6.0), (16, 12, 128, 6.0), (16, 12, 129, 6.0)]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("mode", ["bottom_wall", "slit"])
@pytest.mark.parametrize("nx,ny,nz,zmax", SHAPES)
def test_tiled_solve_at_the_edges_matches_oracle(nx, ny, nz, zmax, mode, precision):
    params = small_params(mode, nx=nx, ny=ny, nz=nz, zmax=zmax, torque=True)
    pos, F, T = random_particles(params, 7, seed=nz)
    U_ref, W_ref = mobility(oracle_params(params), pos, F, T)
    U, W = gpu_mobility(params, pos, F, T, precision)
    assert rel_l2(U, U_ref) <= TOL[precision]
    assert rel_l2(W, W_ref) <= TOL[precision]
