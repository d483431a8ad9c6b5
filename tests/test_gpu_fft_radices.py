"""Every radix of the xy transforms (2 to 16, composite ones among them) in every pass variant that fits,
against the oracle at the parity bars: 210 = 15 x 14, 90 = 10 x 9, 126 = 14 x 9, 225 = 15 x 15, 150 = 15 x 10,
36 = 6 x 6, 98 = 14 x 7, 96 = 12 x 8."""

import pytest

from gpu_helpers import gpu_mobility, oracle_params, rel_l2, small_params
from oracle.stokes import mobility
from paper_2210_01837_gb300 import binding
from paper_2210_01837_gb300.workloads import random_particles

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-9, "mixed": 1e-5}


@pytest.mark.parametrize("nx,ny", [(210, 36), (36, 210), (126, 90), (90, 126), (150, 98), (96, 225)])
def test_every_radix_in_every_variant_matches_oracle(nx, ny):
    params = small_params("bottom_wall", nx=nx, ny=ny, nz=13, zmax=4.0, torque=True)
    pos, F, T = random_particles(params, 12, seed=nx + ny)
    U_ref, W_ref = mobility(oracle_params(params), pos, F, T)
    for precision in ("fp64", "mixed"):
        plan = binding.Plan.from_params(params, with_torque=True, precision=precision, max_n=len(pos))
        tried = 0
        for rows in (0, 1):
            for cols in (0, 1, 2, 3):
                for width in (1, 2, 4, 8):
                    try:
                        plan.set_fft(rows, cols, width)
                    except binding.DpsError:
                        continue  # the shape does not fit
                    tried += 1
                    U, W = gpu_mobility(params, pos, F, T, precision, plan=plan)
                    assert rel_l2(U, U_ref) <= TOL[precision], (precision, rows, cols, width)
                    assert rel_l2(W, W_ref) <= TOL[precision], (precision, rows, cols, width)
        assert tried >= 8
        plan.close()


@pytest.mark.parametrize("nx", [
    3136, 3584,  # last stage 14 (float rows' default there), first 16
    1600, 2240,  # last stage 10
    384,         # last stage 6
    896, 1344,   # first stage 14
    640,         # first stage 10
])
def test_paired_first_and_last_stages_match_oracle(nx):
    """Register-staged rows whose last stage splits the half spectra and whose first stage joins them in
    registers: spans that are multiples of 32, at the composite radices; an odd row count leaves one row
    without a partner."""
    params = small_params("bottom_wall", nx=nx, ny=15, nz=9, zmax=4.0, torque=True)
    pos, F, T = random_particles(params, 12, seed=nx)
    U_ref, W_ref = mobility(oracle_params(params), pos, F, T)
    for precision in ("fp64", "mixed"):
        plan = binding.Plan.from_params(params, with_torque=True, precision=precision, max_n=len(pos))
        info = plan.info()
        if precision == "mixed" and nx >= 3136:
            assert info.fft_register_rows == 1
        plan.set_fft(1, info.fft_register_cols, info.fft_col_width)
        U, W = gpu_mobility(params, pos, F, T, precision, plan=plan)
        plan.close()
        assert rel_l2(U, U_ref) <= TOL[precision], precision
        assert rel_l2(W, W_ref) <= TOL[precision], precision


@pytest.mark.parametrize("n", [3430, 3528, 3600, 3840])
def test_longest_double_sizes_match_oracle(n):
    """Double rows and columns that only the composite radices fit (3840 = 16 16 15 in 256 threads), in every
    variant that they have."""
    for nx, ny in ((n, 16), (16, n)):
        params = small_params("bottom_wall", nx=nx, ny=ny, nz=9, zmax=4.0, torque=True)
        pos, F, T = random_particles(params, 12, seed=n)
        U_ref, W_ref = mobility(oracle_params(params), pos, F, T)
        plan = binding.Plan.from_params(params, with_torque=True, precision="fp64", max_n=len(pos))
        info = plan.info()
        for cols in (info.fft_register_cols,) if nx == n else (1, 2, 3):
            try:
                plan.set_fft(info.fft_register_rows, cols, info.fft_col_width)
            except binding.DpsError:
                assert cols != info.fft_register_cols
                continue
            U, W = gpu_mobility(params, pos, F, T, "fp64", plan=plan)
            assert rel_l2(U, U_ref) <= TOL["fp64"], (nx, ny, cols)
            assert rel_l2(W, W_ref) <= TOL["fp64"], (nx, ny, cols)
        plan.close()
