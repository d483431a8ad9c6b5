"""The envelope records: particle counts on both sides of every switch of the particles per block (1 to 32), a last
block that is not full, one and two record heads, the derivative slab, and particles that are refused.  The
velocities of the first particles must not depend on force-free particles behind them, which change the blocks
but not the flow (1e-12 in double: the same sums over another bin order; 1e-6 mixed)."""

import numpy as np
import pytest

from gpu_helpers import gpu_mobility, rel_l2, small_params, to_dev
from paper_2210_01837_gb300 import binding
from paper_2210_01837_gb300.workloads import random_particles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("route", [False, "spectral_curl", "kernel_derivative"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_velocities_do_not_depend_on_force_free_neighbours(route, precision):
    params = small_params("slit", nx=72, ny=60, nz=33, torque=bool(route))
    counts = [1, 7, 303, 304, 607, 608, 609, 1217, 2433, 4865, 9729, 49151, 49157]
    pos, F, T = random_particles(params, counts[-1], seed=11)
    if not route:
        T = None
    F[1:] = 0.0
    if route:
        T[1:] = 0.0
    with_torque = route if route else False
    plan = binding.Plan.from_params(params, with_torque=with_torque, precision=precision, max_n=len(pos))
    bar = 1e-12 if precision == "fp64" else 1e-6
    ref = gpu_mobility(params, pos, F, T, precision, plan=plan)
    for n in counts:
        got = gpu_mobility(params, pos[:n], F[:n], T[:n] if route else None, precision, plan=plan)
        assert rel_l2(got[0], ref[0][:n]) <= bar, n
        if route:
            assert rel_l2(got[1], ref[1][:n]) <= bar, n
    plan.close()


@pytest.mark.parametrize("n,bad", [(1, 0), (40, 39), (5000, 33)])
def test_refused_particles_are_reported(n, bad):
    params = small_params("bottom_wall", nx=72, ny=60, nz=33, torque=True)
    pos, F, T = random_particles(params, n, seed=n)
    plan = binding.Plan.from_params(params, with_torque=True, precision="mixed", max_n=n)
    for what, want in ((np.nan, binding.DPS_ERR_NONFINITE), (params["zmax"], binding.DPS_ERR_OUT_OF_DOMAIN)):
        p = pos.copy()
        p[bad, 2] = what
        plan.apply(to_dev(p), to_dev(F), to_dev(T))
        assert plan.status() == want
    plan.apply(to_dev(pos), to_dev(F), to_dev(T))
    assert plan.status() == binding.DPS_OK
    plan.close()
