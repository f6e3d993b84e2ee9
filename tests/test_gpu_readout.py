"""The fields of states that the healthy range does not meet: densities that cancel to
almost nothing, populations that are subnormal, huge, infinite or NaN.  rho' is exact, so
the velocity is the quotient (rho0 u0 + j') / (rho0 + rho') of known numbers."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6350_gb300 import lbm

    lbm.load()


def _check(got, num, rho):
    """Within one unit in the last place of the correctly rounded quotient: the kernels
    round it correctly but for ties that their remainder cannot tell apart."""
    with np.errstate(all="ignore"):
        want = num / rho
    finite = np.isfinite(want)
    np.testing.assert_array_equal(np.where(finite, 0.0, got), np.where(finite, 0.0, want))
    off = np.abs(got[finite] - want[finite])
    assert np.all(off <= np.spacing(np.abs(want[finite]))), off.max()
    np.testing.assert_array_equal(got[want == 0.0], want[want == 0.0])


# rho0 that FP32 holds exactly, and such that it does not
@pytest.mark.parametrize("rho0", [1.0, 1.1, 0.3, 7.7])
@pytest.mark.parametrize("u0", [0.0, 0.11])
def test_velocity_where_the_density_cancels(rho0, u0):
    """Two populations per column, uniform along y: the rest one carries the density, the
    one moving along y the momentum."""
    from paper_1203_6350_gb300 import lbm

    with np.errstate(over="ignore"):
        rest = [-rho0 * (1.0 - k) for k in (1e-2, 5e-4, 1e-5, 1e-6, 3e-7, 1e-7, 5e-8, 0.0, -1e-7)]
        rest += [0.0, 1e-44, 1e-3, -2.0 * rho0, 1e18, 3e38, np.inf, -np.inf, np.nan]
        move = [0.0, 1e-45, 1e-30, 1e-8, 0.013, -0.4, 1e25, -np.inf, np.nan]
        a, b = (v.ravel() for v in np.meshgrid(np.float32(rest), np.float32(move)))
    nx, ny = a.size, 4
    with lbm.Lattice(nx, ny, "f32", rho0, (0.0, u0), 1.9, bc="periodic") as lat:
        state = np.zeros((9, ny, lat.state_bytes() // (36 * ny)), dtype=np.float32)
        state[0, :, :nx] = a
        state[2, :, :nx] = b
        lat.set_state(state.view(np.uint8).ravel(), 0)
        dr, _, uy = lat.moments()
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(dr[1], (a + b).astype(np.float64))
        fma = [float(Fraction(rho0) * Fraction(u0) + Fraction(float(v))) if np.isfinite(v)
               else float(v) for v in b]  # rho0 u0 + j', rounded once
        _check(uy[1], np.array(fma), rho0 + dr[1])
