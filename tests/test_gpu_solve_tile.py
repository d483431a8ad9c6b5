"""The tiled solve at the edges of its ranges: fewest and most nodes, even and odd node counts (parities
of unequal length, rows short of whole batches), boxes whose wavenumbers end inside a tile or fill fewer
tiles than a block, odd sizes without Nyquist columns, and the first node count past it; each against
the oracle at the parity bars (1e-9 in double, 1e-5 in mixed precision)."""

import numpy as np
import pytest

from oracle.stokes import mobility
from paper_2210_01837_gb300 import binding
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


# slip lengths and wall velocities: the wall rows of k = 0 as well as those of every other wavenumber
WALLS = dict(slip_bottom=0.4, slip_top=0.7, uw_bottom=(0.3, -0.2), uw_top=(-0.5, 0.6))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny,nz,zmax", [(27, 25, 34, 6.0), (40, 36, 33, 6.0)])
def test_one_block_runs_all_tiles_and_the_zero_mode(nx, ny, nz, zmax, precision):
    """22 and 48 tiles in one block: the rings of constants (16 tiles) and of wall values (9) wrap, and the
    zero mode, on a warp between two of its tiles, takes that warp's shared memory for a while.  The
    wavenumbers are independent, so the result is that of the default grid bit for bit."""
    params = small_params("slit", nx=nx, ny=ny, nz=nz, zmax=zmax, torque=True)
    params.update(WALLS)
    pos, F, T = random_particles(params, 9, seed=nx)
    U_ref, W_ref = mobility(oracle_params(params), pos, F, T)
    plan = binding.Plan.from_params(params, with_torque=True, precision=precision, max_n=len(pos))
    U0, W0 = gpu_mobility(params, pos, F, T, precision, plan=plan)
    plan.set_pipeline(1, 1)
    U1, W1 = gpu_mobility(params, pos, F, T, precision, plan=plan)
    plan.close()
    assert rel_l2(U0, U_ref) <= TOL[precision]
    assert rel_l2(W0, W_ref) <= TOL[precision]
    assert (U1 == U0).all() and (W1 == W0).all()


@pytest.mark.parametrize("nz", [33, 97])
@pytest.mark.parametrize("torque", [True, False])
def test_overflow_is_never_a_finite_wrong_number(nz, torque):
    """Forces of 1e37 overflow the float spectra: what comes out is not finite, or right at the parity bar."""
    params = small_params("slit", nx=40, ny=36, nz=nz, zmax=8.0, torque=torque)
    pos, F, T = random_particles(params, 20, seed=3, torques=torque)
    T = None if T is None else 0.0 * T
    U_ref, _ = mobility(oracle_params(params), pos, F, T)
    U, _ = gpu_mobility(params, pos, 1e37 * F, T, "mixed")
    finite = np.isfinite(U)
    assert np.all(np.abs(U[finite] / 1e37 - U_ref[finite]) <= TOL["mixed"] * np.abs(U_ref).max())


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("mode", ["bottom_wall", "slit"])
@pytest.mark.parametrize("nx,ny,nz,zmax", SHAPES + [(16, 12, 126, 6.0), (16, 12, 127, 6.0)])
def test_wall_conditions_at_the_edges_match_oracle(nx, ny, nz, zmax, mode, precision):
    """Slip and wall velocities take more shared memory and a longer table row: the last node counts whose
    block fits (126 in double) and the first that take the thread-per-wavenumber solve."""
    params = small_params(mode, nx=nx, ny=ny, nz=nz, zmax=zmax, torque=True)
    params.update({k: v for k, v in WALLS.items() if mode == "slit" or k.endswith("bottom")})
    pos, F, T = random_particles(params, 7, seed=nz)
    U_ref, W_ref = mobility(oracle_params(params), pos, F, T)
    U, W = gpu_mobility(params, pos, F, T, precision)
    assert rel_l2(U, U_ref) <= TOL[precision]
    assert rel_l2(W, W_ref) <= TOL[precision]
