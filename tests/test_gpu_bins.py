"""Binning at the sizes where a bin's list changes hands in the sort: bins of 0, 1, 2, 31 to 33, 255 to 257
particles (257 keeps the scatter's order) in one call.  Repeated products agree bit for bit while no bin is
above 256, and every product agrees with the oracle."""

import numpy as np
import pytest

from gpu_helpers import gpu_mobility, oracle_params, rel_l2, small_params
from oracle.stokes import mobility
from paper_2210_01837_gb300 import binding

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-9, "mixed": 1e-5}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("counts", [(1, 2, 31, 32, 33, 0, 255, 256), (257, 64, 0, 3, 300, 1, 96, 2)])
def test_bins_of_every_size_are_ordered(counts, precision):
    params = small_params("bottom_wall", nx=64, ny=32, nz=17, zmax=6.0, torque=True)  # 2 x 4 bins of 32 x 8 nodes
    h = params["Lx"] / params["nx"]
    rng = np.random.default_rng(sum(counts))
    pos = []
    for b, c in enumerate(counts):
        x0, y0 = 32 * h * (b % 2), 8 * h * (b // 2)
        pos.append(np.stack([rng.uniform(x0, x0 + 32 * h, c), rng.uniform(y0, y0 + 8 * h, c), rng.uniform(1.0, 3.5, c)], 1))
    pos = np.concatenate(pos)
    pos = pos[rng.permutation(len(pos))]  # bins interleaved, as a caller's particles come
    F, T = rng.standard_normal(pos.shape), rng.standard_normal(pos.shape)
    U_ref, W_ref = mobility(oracle_params(params), pos, F, T)
    plan = binding.Plan.from_params(params, with_torque=True, precision=precision, max_n=len(pos))
    runs = [gpu_mobility(params, pos, F, T, precision, plan=plan) for _ in range(4)]
    plan.close()
    for U, W in runs:
        assert rel_l2(U, U_ref) <= TOL[precision]
        assert rel_l2(W, W_ref) <= TOL[precision]
        if max(counts) <= 256:
            assert np.array_equal(U, runs[0][0]) and np.array_equal(W, runs[0][1])
