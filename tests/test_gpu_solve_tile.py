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


# (mode, precision, nx, ny, nz, tiled): either side of the lines of the rule
ROUTES = [("free", "mixed", 240, 240, 81, True), ("free", "mixed", 256, 240, 81, False),
          ("free", "fp64", 240, 240, 66, True), ("free", "fp64", 256, 240, 66, False),
          ("slit", "mixed", 320, 320, 81, True), ("slit", "mixed", 324, 324, 81, False),
          ("bottom_wall", "fp64", 320, 320, 66, True), ("bottom_wall", "fp64", 324, 324, 66, False),
          ("free", "mixed", 336, 336, 65, True), ("slit", "mixed", 384, 384, 24, False),
          ("slit", "mixed", 384, 384, 25, True), ("bottom_wall", "mixed", 840, 840, 32, False),
          ("bottom_wall", "mixed", 840, 840, 33, True), ("free", "fp64", 840, 840, 33, False),
          ("free", "fp64", 800, 800, 33, True)]


@pytest.mark.parametrize("mode,precision,nx,ny,nz,tiled", ROUTES)
def test_either_side_of_the_rule_matches_the_general_solve(mode, precision, nx, ny, nz, tiled, monkeypatch):
    """The chosen solve against the one that factorises as it goes and takes every plan; which one was
    chosen shows in the grid (one block of 128 wavenumbers each, or fewer tiles' blocks)."""
    params = small_params(mode, nx=nx, ny=ny, nz=nz, zmax=7.0, torque=False)
    pos, F, _ = random_particles(params, 40, seed=nz, torques=False)
    plan = binding.Plan.from_params(params, with_torque=False, precision=precision, max_n=len(pos))
    blocks = plan.info().solve_blocks
    U, _ = gpu_mobility(params, pos, F, None, precision, plan=plan)
    plan.close()
    monkeypatch.setenv("DPS_SOLVE_TABLE", "0")
    general = binding.Plan.from_params(params, with_torque=False, precision=precision, max_n=len(pos))
    assert (blocks < general.info().solve_blocks) == tiled
    U_ref, _ = gpu_mobility(params, pos, F, None, precision, plan=general)
    general.close()
    assert rel_l2(U, U_ref) <= TOL[precision]


@pytest.mark.parametrize("nx,ny,nz,precision", [(384, 384, 65, "mixed"), (40, 36, 33, "fp64"), (16, 12, 8, "mixed")])
def test_every_grid_of_the_thread_per_wavenumber_solve_is_accepted(nx, ny, nz, precision, monkeypatch):
    """Grids set for that solve (three blocks an SM, or all wavenumbers' blocks) hold for the tiled one too,
    which may choose fewer; blocks without a tile leave the result as it is."""
    params = small_params("slit", nx=nx, ny=ny, nz=nz, zmax=6.0, torque=False)
    pos, F, _ = random_particles(params, 9, seed=nz, torques=False)
    kw = dict(with_torque=False, precision=precision, max_n=len(pos))
    monkeypatch.setenv("DPS_SOLVE_TABLE", "0")
    general = binding.Plan.from_params(params, **kw)
    most = general.info().solve_blocks
    general.close()
    monkeypatch.delenv("DPS_SOLVE_TABLE")
    plan = binding.Plan.from_params(params, **kw)
    own = plan.info().solve_blocks
    U0, _ = gpu_mobility(params, pos, F, None, precision, plan=plan)
    for blocks in {most, max(1, most // 2), own}:
        plan.set_pipeline(blocks, 1)
        U, _ = gpu_mobility(params, pos, F, None, precision, plan=plan)
        assert (U == U0).all()
    with pytest.raises(binding.DpsError):
        plan.set_pipeline(max(most, own) + 1, 1)
    plan.close()
