"""Which kernels a lattice or a batch takes by default, by size, layer and storage, and that
the results do not depend on it."""
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


def _ramp(n, width, chi=0.3):
    i = np.arange(n)
    d = np.clip(width - np.minimum(i, n - 1 - i), 0, width) / max(width, 1)
    return chi * d * d


def _lattice(nx, ny, bc, storage, variant, width):
    from paper_1203_6350_gb300 import lbm

    lat = lbm.Lattice(nx, ny, storage, 1.0, (0.04, -0.02), 1.6, bc=bc)
    lat.set_sponge(variant, _ramp(nx, width), _ramp(ny, width))
    lat.init_pulse(1e-3, 9.0, 0.4 * nx, 0.6 * ny)
    return lat


def _marches(lat):
    from paper_1203_6350_gb300 import lbm

    return lbm.lbm_step_launches(lat.h, 12) < 12 // lat.steps_per_launch or (
        lat.storage != "f32" and lat.steps_per_launch == 2)


# (shape, boundary, storage, variant, layer, marching)
ROUTES = [((1024, 1024), "dirichlet", "bf16dev", "II", 64, True),
          ((1024, 1024), "dirichlet", "bf16dev", "II", 511, False),
          ((850, 1054), "dirichlet", "f16dev", "I", 250, False),
          ((1024, 1024), "dirichlet", "f16dev", "none", 0, True),
          ((1024, 1024), "dirichlet", "f32", "II", 511, True),
          ((1344, 1093), "periodic", "f16dev", "III", 20, True),
          ((1344, 1093), "periodic", "f16dev", "III", 545, False),
          ((8640, 151), "periodic", "bf16dev", "none", 0, False),
          ((11532, 139), "dirichlet", "f16dev", "none", 0, False),
          ((1401, 1405), "periodic", "f32", "II", 20, True),
          ((1401, 1405), "periodic", "f32", "III", 699, False),
          ((1401, 1405), "periodic", "f16dev", "II", 20, False),
          ((1403, 1405), "periodic", "bf16dev", "none", 0, False),
          ((1152, 1151), "periodic", "f32", "I", 500, True)]


@pytest.mark.parametrize("shape,bc,storage,variant,width,marching", ROUTES)
def test_marching_is_taken_where_it_is_faster(shape, bc, storage, variant, width, marching):
    with _lattice(*shape, bc, storage, variant, width) as lat:
        assert _marches(lat) == marching
        lat.step(14)
        got, _ = lat.get_state()
    with _lattice(*shape, bc, storage, variant, width) as lat:
        lat.steps_per_launch = lat.steps_per_launch
        assert not _marches(lat)
        lat.step(14)
        np.testing.assert_array_equal(got, lat.get_state()[0])


def test_the_choice_follows_the_layer_until_a_kernel_is_named():
    nx = ny = 1024
    thick, thin = _ramp(nx, 500), _ramp(nx, 40)
    with _lattice(nx, ny, "dirichlet", "bf16dev", "II", 500) as lat:
        lat.step(70)
        lat.set_sponge("II", thin, thin)
        assert _marches(lat)
        lat.step(70)
        lat.set_sponge("III", thick, thick)
        assert not _marches(lat)
        lat.step(5)
        got, _ = lat.get_state()
    with _lattice(nx, ny, "dirichlet", "bf16dev", "II", 500) as lat:
        lat.steps_per_launch = 1  # (named while the choice was this one already)
        lat.step(70)
        lat.set_sponge("II", thin, thin)
        assert not _marches(lat)
        lat.step(70)
        lat.set_sponge("III", thick, thick)
        lat.step(5)
        np.testing.assert_array_equal(got, lat.get_state()[0])
