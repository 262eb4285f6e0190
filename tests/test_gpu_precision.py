"""Stated precision bounds of the float paths against FP64 (Example 3, exact solution)."""
import math

import numpy as np
import pytest

import exact
import oracle
from gpucase import Case
from paper_1909_13263_gb300 import inputs, native

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    native.load()
    native.use_torch_allocator(True)
    yield


def _solve(n, precision):
    x, dx = inputs.axis(n, -2.0, 2.0, "periodic")
    tf = 0.5 / math.pi**2
    with native.Solver(dim=2, nx=n, ny=n, xlo=-2.0, xhi=2.0, ylo=-2.0, yhi=2.0, ham="burgers2d",
                       precision=precision) as s:
        s.set_phi0(inputs.phi0_negcos_diag_2d(x, x))
        s.step_to(tf)
        return np.abs(s.get_phi() - exact.negcos_diag_2d("burgers2d", x, x, tf)).mean()


@pytest.mark.parametrize("n", [80, 160])
def test_mixed_l1_within_105_percent_of_fp64_where_discretisation_dominates(n):
    e64, emx = _solve(n, "fp64"), _solve(n, "mixed")
    assert emx <= 1.05 * e64, (emx, e64)


def test_mixed_beats_fp32_by_orders_of_magnitude_on_fine_grids():
    e64, emx, e32 = _solve(400, "fp64"), _solve(400, "mixed"), _solve(400, "fp32")
    assert emx < 2.0 * e64 and e32 > 20.0 * emx, (e64, emx, e32)


# Where phi_x = phi_y = 0 Burgers' H is 1/2, and with a time step of 2^-6 every stage of Step 5 is exact in float:
# the change over a step is -2^-7 to the last bit (up to the float 2/3 and 1/3 of stage 3, half a unit of the
# increment or of phi).  A rounding bias of H, however small, shows here at full size and would grow with t.
@pytest.mark.parametrize("precision", ["mixed", "fp32"])
@pytest.mark.parametrize("alpha_mode", ["global_lagged", "local_lagged", "fixed"])
def test_burgers_hamiltonian_is_unbiased_on_constants(precision, alpha_mode):
    value, dt, steps = 0.25, 2.0**-6, 8
    fixed = (1.0, 1.0) if alpha_mode == "fixed" else (0.0, 0.0)
    with native.Solver(dim=2, nx=70, ny=40, xlo=-2.0, xhi=2.0, ylo=-2.0, yhi=2.0, ham="burgers2d", precision=precision,
                       alpha_mode=alpha_mode, alpha_fixed=fixed) as s:
        s.set_phi0(np.full((40, 70), value))
        for _ in range(steps):
            s.run_stage(1, dt)
            if _ == 0:
                np.testing.assert_array_equal(s.get_stage_phi(1), value - dt / 2)
            s.run_stage(2, dt)
            s.run_stage(3, dt)
        err = np.abs(s.get_phi() - (value - steps * dt / 2)).max()
    unit = dt / 2 if precision == "mixed" else value
    assert err <= steps * unit * 2.0**-24


# The rounding of a smooth H must not lean to one side: over a line of 8192 nodes the mean error of L, from the first
# stage's increment against the oracle, stays below a tenth of the last place of the derivatives' sum (2^-22 for sums
# up to 4, here pi); errors that fall at random average to a hundredth.
@pytest.mark.parametrize("theta", [0.0, 0.3, 1.1, 2.0])
def test_mixed_rounding_of_smooth_data_is_unbiased(theta):
    case = Case(2, 8192, 32, "burgers2d", precision="mixed", lo=-2.0, hi=2.0, alpha_mode="fixed", alpha_fixed=(2.5, 2.5))
    x, _ = inputs.axis(8192, -2.0, 2.0, "periodic")
    phi = np.tile(-np.cos(0.5 * math.pi * x + theta), (32, 1))
    dt = 2.0**-13
    with case.solver() as s:
        s.set_phi0(phi)
        s.run_stage(1, dt)
        L = (s.get_stage_phi(1) - s.get_phi()) / dt
    err = L - oracle.L_of(case.cfg(), phi, np.array([2.5, 2.5]))
    assert abs(err.mean()) <= 0.1 * 2.0**-22
