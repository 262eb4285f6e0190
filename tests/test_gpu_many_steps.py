"""2D float solves whose RK3 steps run several to a launch, against the same steps made of single stages.

Both run the same arithmetic on the same tiles, so every result is bitwise the same: the field, the grid
maxima and the time.
"""
import numpy as np
import pytest

from gpucase import Case
from paper_1909_13263_gb300 import native

pytestmark = pytest.mark.gpu

# one tile, tile edges crossed by one node, fewer nodes than a stencil is wide, ragged, more tiles than CTAs
SHAPES = [(64, 32), (65, 33), (5, 4), (127, 95), (1500, 901)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    native.load()
    native.use_torch_allocator(True)
    yield


def _case(shape, precision="mixed", weights="arclength", alpha_mode="global_lagged", ham="burgers2d"):
    return Case(2, *shape, ham, precision=precision, weights=weights, alpha_mode=alpha_mode,
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
                                  dict(alpha_mode="fixed"), dict(ham="eikonal2d", precision="fp32")], ids=str)
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
