"""Time 0: the device-built pulse against the same field handed over as an array,
at the edges of the pulse kernel's blocks (128 columns, up to 64 rows)."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

# the field's density is rounded at 1 (2^-53) before its deviation is taken, which may
# turn the rounding to the storage format: one unit in the last place at the largest value
ULP = {"f64": 2.0**-40, "f32": 2.0**-22, "f16dev": 2.0**-10, "bf16dev": 2.0**-7}
DTYPE = {"f64": np.float64, "f32": np.float32, "f16dev": np.float16}


def _values(buf, storage):
    if storage == "bf16dev":
        return (buf.view(np.uint16).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    return buf.view(DTYPE[storage]).astype(np.float64)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6350_gb300 import lbm

    lbm.load()


@pytest.mark.parametrize("shape", [(2, 1), (3, 5), (128, 64), (129, 65), (257, 3), (1500, 1301)])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic", "channel"])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev", "bf16dev"])
def test_the_pulse_is_the_field_it_describes(shape, bc, storage):
    from paper_1203_6350_gb300 import lbm

    nx, ny = shape
    eps, b, x0, y0 = 1e-3, 6.0, 0.4 * nx, 0.7 * ny
    u0 = (0.05, -0.02)
    dr = wl.gaussian_pulse(nx, ny, x0, y0, eps, b)
    with lbm.Lattice(nx, ny, storage, 1.0, u0, 1.9, bc=bc) as lat:
        lat.init_pulse(eps, b, x0, y0)
        got = _values(lat.get_state()[0], storage)
        lat.init_equilibrium(1.0 + dr, np.full_like(dr, u0[0]), np.full_like(dr, u0[1]))
        want = _values(lat.get_state()[0], storage)
    assert np.abs(got - want).max() <= ULP[storage] * np.abs(want).max()


def test_a_pulse_narrower_than_any_number():
    """alpha = ln 2 / b^2 overflows: the density is the far field at every cell."""
    from paper_1203_6350_gb300 import lbm

    with lbm.Lattice(40, 30, "f32", 1.0, (0.0, 0.0), 1.9) as lat:
        lat.init_pulse(1e-3, 1e-170, 10.5, 10.5)
        assert not _values(lat.get_state()[0], "f32").any()
