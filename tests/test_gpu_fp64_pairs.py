"""FP64 stages whose nonlinear weights are formed in float pairs, against the FP64 oracle.

On smooth data every segment qualifies for the pairs.  Kernel and oracle then differ by rounding only: a
stage rounds phi + dt L once (half a unit of the largest |phi|, u = 2^-53) after three or four rounded
operations of the same size, and L's own error, a few u of |phi_x|, enters times dt |H_p| <= 0.6 dx; the
bound is 16 u of max |phi|.  Data with kinks, noise or an offset mix qualifying and other segments; there
the indicators of single-precision size are amplified as in test_gpu_parity.py (1e-12).
"""
import math

import numpy as np
import pytest

import oracle
from gpucase import Case, oracle_stages, rel_err
from paper_1909_13263_gb300 import inputs, native

pytestmark = pytest.mark.gpu

SMOOTH_TOL = 16 * 2.0**-53
FP64_TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _lib():
    native.load()
    native.use_torch_allocator(True)
    yield


def _errors(case, phi0):
    a, _ = oracle.alpha_of(case.cfg(), phi0)
    dt = 0.6 / (a[0] / case.dx + (a[1] / case.dy if case.dim == 2 else 0.0))
    ref = oracle_stages(case, phi0, dt)
    with case.solver() as s:
        s.set_phi0(phi0)
        errs = []
        for stage in (1, 2, 3):
            s.run_stage(stage, dt)
            errs.append(rel_err(s.get_stage_phi(stage) if stage < 3 else s.get_phi(), ref[stage - 1]))
    return errs


def _smooth(case):
    # one wave over the domain, resolved by the smallest of the grids below
    x, _ = inputs.axis(case.nx, case.lo, case.hi, case.bc)
    if case.dim == 1:
        return -np.cos(np.pi * x + 0.3)
    y, _ = inputs.axis(case.ny, case.lo, case.hi, case.bc)
    return -np.cos(np.pi * (x[None, :] + 2.0 * y[:, None]) / 2.0 + 0.3)


# edges of the 16 x 16 and 32 x 16 tiles and of the 1D tiles, ragged and rectangular
@pytest.mark.parametrize("weights", ["arclength", "jp"])
@pytest.mark.parametrize("shape", [(2, 31, 33), (2, 64, 48), (2, 161, 163), (2, 1025, 130), (1, 63, 1), (1, 64, 1),
                                   (1, 65, 1), (1, 321, 1), (1, 5000, 1)], ids=str)
def test_smooth_stages_match_oracle_to_rounding(shape, weights):
    dim, nx, ny = shape
    case = Case(dim, nx, ny, "negcos2d" if dim == 2 else "burgers1d", weights=weights, lo=-2.0 if dim == 2 else -1.0,
                hi=2.0 if dim == 2 else 1.0, alpha_mode="global_lagged" if dim == 2 else "local_lagged")
    assert max(_errors(case, _smooth(case))) <= SMOOTH_TOL


@pytest.mark.parametrize("weights", ["arclength", "jp"])
@pytest.mark.parametrize("kind", ["kinks", "noise", "offset", "huge", "tiny"])
def test_mixed_segments_match_oracle(kind, weights):
    case = Case(2, 97, 75, "sin2d", bc="linextrap", weights=weights)
    x, _ = inputs.axis(97, -1.0, 1.0, "linextrap")
    y, _ = inputs.axis(75, -1.0, 1.0, "linextrap")
    phi0 = math.pi * (np.abs(y[:, None] - 0.03) - np.abs(x[None, :] + 0.01))
    if kind == "noise":
        phi0[20:30, 40:60] += 0.01 * inputs.random_field(10, 20, 3, "rough")
    elif kind == "offset":
        phi0 = 1e3 + np.sin(2.0 * x[None, :] + y[:, None])
    elif kind == "huge":
        case.ham, phi0 = "burgers2d", phi0 * 1e5
    elif kind == "tiny":
        case.ham, phi0 = "burgers2d", phi0 * 1e-40
    assert max(_errors(case, phi0)) <= FP64_TOL


# 1D grids that run whole steps in one launch (up to 1024 nodes): edges of the shares of 1, 2, 4 and 8 CTAs
@pytest.mark.parametrize("nx", [2, 5, 64, 65, 128, 129, 257, 513, 1024, 1025])
@pytest.mark.parametrize("kw", [dict(bc="periodic"), dict(bc="linextrap", alpha_mode="global_lagged"),
                                dict(bc="periodic", weights="jp", alpha_mode="fixed", alpha_fixed=(5.0, 0.0)),
                                dict(bc="linextrap", dt_mode="dx53")], ids=lambda k: "-".join(map(str, k.values())))
def test_line_solve_matches_oracle(nx, kw):
    case = Case(1, nx, 1, "burgers1d", **{"alpha_mode": "local_lagged", **kw})
    x, _ = inputs.axis(nx, -1.0, 1.0, case.bc)
    phi0 = -np.cos(np.pi * x + 0.3) + 0.2 * np.abs(x)
    a, _ = oracle.alpha_of(case.cfg(), phi0)
    alpha = case.alpha_fixed[0] if case.alpha_mode == "fixed" else a[0]
    tf = 7.5 * 0.6 * (case.dx ** (5.0 / 3.0) if case.dt_mode == "dx53" else case.dx) / alpha
    ref, steps_ref, t_ref, _, st = oracle.solve(case.cfg(), phi0, tf)
    assert st == 0
    with case.solver() as s:
        s.set_phi0(phi0)
        n = s.step_to(0.4 * tf)
        mid, state = s.get_phi(), s.get_state()
        n += s.step_to(tf)
        whole, end = s.get_phi(), s.get_state()
        # resumed from the state in between: the same bits
        s.set_state(state, mid)
        s.step_to(tf)
        assert np.array_equal(s.get_phi(), whole)
        # the same number of steps without clipping, then one per-stage step on top of it
        s.set_phi0(phi0)
        s.advance(3)
        s.advance(2)
        five = s.get_phi()
        s.set_phi0(phi0)
        s.advance(5)
        assert np.array_equal(s.get_phi(), five)
        assert s.get_state().steps == 5
    assert end.t == t_ref == tf
    # one extra step at most where the run was stopped in between
    assert steps_ref <= n <= steps_ref + 1
    with case.solver() as s:
        s.set_phi0(phi0)
        assert s.step_to(tf) == steps_ref
        assert rel_err(s.get_phi(), ref) <= FP64_TOL


def test_line_solve_reports_nonfinite():
    case = Case(1, 200, 1, "burgers1d", alpha_mode="local_lagged")
    phi0 = case.field(seed=2, kind="smooth")
    with case.solver() as s:
        s.set_phi0(phi0)
        s.advance(1)
        bad = s.get_phi()
        bad[77] = np.nan
        s.set_state(s.get_state(), bad)
        with pytest.raises(native.AlwError) as e:
            s.step_to(1.0)
        assert e.value.status == native.ENONFINITE
        assert s.get_state().steps == 1


# Jiang-Peng indicators far below one: q = (eps + 13 d^2 + 3 e^2)^2 reaches and passes the smallest float, down to
# where only double holds it.  H is linear in the derivatives to first order (advection, sin(p + q)), so that phi
# keeps the size of the data.
@pytest.mark.parametrize("eps, size", [(1e-24, 1e-10), (1e-24, 1e-12), (1e-40, 1e-11), (1e-40, 5e-13), (1e-30, 3e-12),
                                       (1e-18, 1e-9), (1e-300, 1e-20)])
@pytest.mark.parametrize("dim, nx", [(1, 80), (1, 320), (1, 2000), (2, 80)])
def test_small_jiang_peng_indicators_match_oracle(dim, nx, eps, size):
    case = Case(dim, nx, 70 if dim == 2 else 1, "sin2d" if dim == 2 else "advect1d", weights="jp", eps=eps, lo=-2.0,
                hi=2.0, alpha_mode="global_lagged" if dim == 2 else "local_lagged")
    phi0 = size * _smooth(case)
    assert max(_errors(case, phi0)) <= FP64_TOL
    # the same step by the solver's own loop (1D: the kernel that runs whole steps)
    a, _ = oracle.alpha_of(case.cfg(), phi0)
    dt = 0.6 / (a[0] / case.dx + (a[1] / case.dy if dim == 2 else 0.0))
    with case.solver() as s:
        s.set_phi0(phi0)
        s.advance(1)
        assert rel_err(s.get_phi(), oracle_stages(case, phi0, dt)[2]) <= FP64_TOL


# Tiles in which many nodes do not qualify are swept in double segment by segment, others node by node.  Noise over
# part of the grid gives both, next to tiles that qualify; grids as above, so that the tile shapes and the ragged
# segments of each are met.
@pytest.mark.parametrize("weights", ["arclength", "jp"])
@pytest.mark.parametrize("nx, ny", [(31, 33), (64, 48), (161, 163), (1025, 130), (600, 611)])
def test_tiles_of_noise_match_oracle(nx, ny, weights):
    case = Case(2, nx, ny, "sin2d", weights=weights, lo=-2.0, hi=2.0)
    phi0 = _smooth(case)
    rough = case.field(seed=8)
    phi0[: ny // 3, : nx // 2] += 0.1 * rough[: ny // 3, : nx // 2]
    scattered = np.random.default_rng(9).random((ny - ny // 2, nx)) < 0.05
    phi0[ny // 2:][scattered] += 0.1 * rough[ny // 2:][scattered]
    assert max(_errors(case, phi0)) <= FP64_TOL


# What the launches of whole steps leave behind (field, ghosts, grid maxima) is what single stages go on from: three
# steps in one launch and one by stages, against four by stages with the same time steps.
@pytest.mark.parametrize("nx", [5, 64, 200, 1024])
@pytest.mark.parametrize("kw", [dict(bc="periodic"), dict(bc="linextrap", alpha_mode="global_lagged"),
                                dict(bc="linextrap", weights="jp", alpha_mode="fixed", alpha_fixed=(5.0, 0.0))],
                         ids=lambda k: "-".join(map(str, k.values())))
def test_stages_go_on_from_a_line_launch(nx, kw):
    case = Case(1, nx, 1, "burgers1d", **{"alpha_mode": "local_lagged", **kw})
    x, _ = inputs.axis(nx, -1.0, 1.0, case.bc)
    phi0 = -np.cos(np.pi * x + 0.3) + 0.2 * np.abs(x)

    def stages(s):
        a = case.alpha_fixed if case.alpha_mode == "fixed" else s.get_state().alpha
        for stage in (1, 2, 3):
            s.run_stage(stage, 0.6 * case.dx / a[0])

    with case.solver() as s, case.solver() as r:
        s.set_phi0(phi0)
        s.advance(3)
        stages(s)
        r.set_phi0(phi0)
        for _ in range(4):
            stages(r)
        assert rel_err(s.get_phi(), r.get_phi()) <= FP64_TOL
        assert s.get_state().alpha[0] == pytest.approx(r.get_state().alpha[0], rel=FP64_TOL)
