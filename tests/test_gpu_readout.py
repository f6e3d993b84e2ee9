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


def _d3_state(lat, shape, planes):
    """The populations of a periodic D3Q15 state that varies along x only."""
    nx, ny, nz = shape
    buf, _ = lat.get_state()
    s = np.zeros((15, nz, ny, buf.nbytes // (15 * nz * ny * 8)))
    for i, v in planes.items():
        s[i, :, :, :nx] = v
    lat.set_state(s.view(np.uint8).ravel(), 0)


def _d3_fields(rho0, planes):
    """(rho', u_y) along x of an FP64 state given by its populations (3: c = +y, 4: -y)."""
    from paper_1203_6350_gb300 import lbm

    shape = (len(planes[0]), 3, 2)
    with lbm.Lattice3(*shape, "f64", rho0, (0.0, 0.0, 0.0), 1.9, bc="periodic") as lat:
        lat.init_equilibrium(np.full(shape[::-1], rho0), 0.0, 0.0, 0.0)
        _d3_state(lat, shape, planes)
        rho, ux, uy, uz = lat.moments()
        return rho[1, 1], ux[1, 1], uy[1, 1], uz[1, 1]


@pytest.mark.parametrize("rho0", [1.0, 3e-18, 5e17])
def test_quotients_of_huge_and_tiny_momenta(rho0):
    """FP64 momenta whose quotient overflows, or whose remainder underflows."""
    j = np.array([0.0, 1.0, -0.3, 1e270, -1e270, 1e300, 1.7e308, -1.7e308, 1e-270, 1e-290,
                  -1e-300, 3e-308, 5e-324, -1e-320])
    rho, ux, uy, uz = _d3_fields(rho0, {0: -j, 3: j})  # the rest population takes it back
    np.testing.assert_array_equal(rho, np.zeros_like(j))
    assert not ux.any() and not uz.any()
    _check(uy, j, np.full_like(j, rho0))


def test_an_infinite_population_leaves_no_velocity():
    """An overflowed cell of a 3-D state: the products of an infinite population with the
    zero components of its velocity are NaN, and so is u.  Finite populations whose sum
    overflows still have the quotient of their momentum."""
    inf, big = np.inf, 1.2e308
    rest = np.array([inf, -inf, np.nan, 0.0, 0.0, 0.0, inf, 0.0, big, big])
    plus = np.array([0.0, 0.0, 0.0, inf, 0.0, np.nan, -inf, inf, 0.0, big])
    minus = np.array([0.0, 0.0, 0.0, 0.0, -inf, 0.0, 0.0, inf, 0.0, 0.0])
    rho, ux, uy, uz = _d3_fields(1.0, {0: rest, 3: plus, 4: minus})
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(rho, rest + plus + minus)
        want = np.full(rest.shape, np.nan)
        want[-2:] = plus[-2:] / (1.0 + rho[-2:])
    np.testing.assert_array_equal(uy, want)
    want[-2:] = 0.0
    np.testing.assert_array_equal(ux, want)
    np.testing.assert_array_equal(uz, want)
