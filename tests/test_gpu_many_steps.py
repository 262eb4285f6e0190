"""2D float solves whose RK3 steps run several to a launch, against the same steps made of single stages.

Both run the same arithmetic on the same tiles, so every result is bitwise the same: the field, the grid
maxima and the time.  The ghosts that the stages extrapolate are checked through the oracle's stages, with the
bound of one float stage (test_gpu_parity.py), restarted at every step from the kernel's own field.
"""
import numpy as np
import pytest

from gpucase import Case, oracle_stages, rel_err
from paper_1909_13263_gb300 import native

pytestmark = pytest.mark.gpu

# one tile, tile edges crossed by one node, fewer nodes than a stencil is wide, ragged, more tiles than CTAs
SHAPES = [(64, 32), (65, 33), (5, 4), (127, 95), (1500, 901)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    native.load()
    native.use_torch_allocator(True)
    yield


def _case(shape, precision="mixed", weights="arclength", alpha_mode="global_lagged", ham="burgers2d",
          bc="periodic"):
    return Case(2, *shape, ham, bc=bc, precision=precision, weights=weights, alpha_mode=alpha_mode,
                alpha_fixed=(2.5, 2.0) if alpha_mode == "fixed" else (0.0, 0.0), lo=-2.0, hi=2.0)


def _phi0(case):
    x = np.linspace(-1.0, 1.0, case.nx, endpoint=False)[None, :]
    y = np.linspace(-1.0, 1.0, case.ny, endpoint=False)[:, None]
    # smooth, with kinks along both directions, and noise in one corner
    phi = np.cos(np.pi * (x + y)) * 0.2 + 0.1 * np.abs(np.sin(np.pi * x)) + 0.1 * np.abs(np.sin(np.pi * y))
    phi[: case.ny // 4, : case.nx // 4] += 1e-3 * case.field()[: case.ny // 4, : case.nx // 4]
    return phi


def _by_stages(case, phi0, steps, stop=None):
    """The steps as single stages; (field, alpha, times), the last step shortened to `stop` steps' end."""
    t, times = 0.0, []
    with case.solver() as s:
        s.set_phi0(phi0)
        for k in range(steps):
            a = case.alpha_fixed if case.alpha_mode == "fixed" else list(s.get_state().alpha)
            dt = 0.6 / (a[0] / case.dx + a[1] / case.dy)
            if stop is not None and k == steps - 1:
                tf = t + stop * dt
                dt, t = tf - t, tf
            else:
                t += dt
            for stage in (1, 2, 3):
                s.run_stage(stage, dt)
            times.append(t)
        return s.get_phi(), list(s.get_state().alpha), times


def _same(s, ref):
    st = s.get_state()
    assert st.steps == len(ref[2]) and st.t == ref[2][-1]
    assert list(st.alpha) == ref[1]
    np.testing.assert_array_equal(s.get_phi(), ref[0])


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("kind", [dict(), dict(precision="fp32"), dict(weights="jp"), dict(alpha_mode="local_lagged"),
                                  dict(alpha_mode="fixed"), dict(ham="eikonal2d", precision="fp32"),
                                  dict(bc="linextrap"), dict(bc="linextrap", precision="fp32")], ids=str)
def test_steps_of_one_launch_equal_single_stages(shape, kind):
    case = _case(shape, **kind)
    phi0 = _phi0(case)
    ref = _by_stages(case, phi0, 4)
    with case.solver() as s:
        for parts in ((4,), (1, 2, 1)):
            s.set_phi0(phi0)
            for n in parts:
                s.advance(n)
            _same(s, ref)
        ref = _by_stages(case, phi0, 4, stop=0.5)
        s.set_phi0(phi0)
        assert s.step_to(ref[2][-1]) == 4
        _same(s, ref)


def test_nonfinite_ends_the_launch_and_is_reported():
    # a fixed alpha of 1e-6 makes the time step several thousand times too long
    case = _case((127, 95), alpha_mode="fixed")
    case.alpha_fixed = (1e-6, 1e-6)
    with case.solver() as s:
        s.set_phi0(_phi0(case))
        s.advance(60)
        with pytest.raises(native.AlwError):
            s.sync()
        s.set_phi0(0.0 * _phi0(case))
        s.advance(3)
        s.sync()
        assert s.get_state().steps == 3


# the last tile two nodes wide and high (the narrowest that extrapolates in the stage), one node (separate ghost
# launches), whole tiles, the smallest grid, more tiles than CTAs
@pytest.mark.parametrize("precision", ["mixed", "fp32"])
@pytest.mark.parametrize("shape", [(66, 34), (65, 34), (66, 33), (128, 64), (2, 2), (1500, 901)], ids=str)
def test_extrapolated_ghosts_match_oracle(shape, precision):
    case = _case(shape, precision=precision, alpha_mode="fixed", ham="sin2d", bc="linextrap")
    case.alpha_fixed = (1.0, 1.0)
    dt = 0.6 / (1.0 / case.dx + 1.0 / case.dy)
    phi = case.field(seed=6)
    with case.solver() as s:
        s.set_phi0(phi)
        errs = []
        for _ in range(3):
            ref = oracle_stages(case, phi, dt)
            for stage in (1, 2, 3):
                s.run_stage(stage, dt)
                phi = s.get_stage_phi(stage) if stage < 3 else s.get_phi()
                errs.append(rel_err(phi, ref[stage - 1]))
    assert max(errs) <= 64 * 2.0**-24, errs


@pytest.mark.parametrize("first_refused", [1, 2, 3])
@pytest.mark.parametrize("how", ["advance", "step_to"])
@pytest.mark.parametrize("kind", ["mixed", "fp32", "line"])
def test_no_room_for_many_steps_returns_to_single_stages(kind, how, first_refused, monkeypatch):
    # a launch of whole steps is refused, at once or in the middle of a call: the stages run one by one from there on
    if kind == "line":
        case = Case(1, 200, 1, "burgers1d", alpha_mode="local_lagged")
        phi0, steps = case.field(seed=4, kind="smooth"), 1200
    else:
        case = _case((127, 95), precision=kind)
        phi0, steps = _phi0(case), 200
    tf = None

    def solve():
        with case.solver() as s:
            s.set_phi0(phi0)
            if how == "advance" or tf is None:
                s.advance(steps)
            else:
                s.step_to(tf)
            phi, st = s.get_phi(), s.get_state()
            s.advance(3)
            s.step_to(s.get_state().t * 1.01)
            s.sync()
            return phi, st.t, st.steps

    tf = solve()[1]
    ref = solve()
    monkeypatch.setenv("ALW_TEST_NO_ROOM_FROM", str(first_refused))
    got = solve()
    if kind == "line":   # the cluster kernel and the stage kernel round differently
        assert got[1] == pytest.approx(ref[1], rel=1e-12) and abs(got[2] - ref[2]) <= 1
        assert rel_err(got[0], ref[0]) <= 1e-12
    else:
        assert got[1:] == ref[1:]
        np.testing.assert_array_equal(got[0], ref[0])
