"""The small-lattice tiles (several steps per launch, the default up to 226^2 cells)
against a launch per step on the same lattices: the stored states agree bit for bit."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6350_gb300 import lbm

    lbm.load()


def _workload(nx, ny, bc, variant, layer, seed):
    rng = np.random.default_rng(seed)

    def profile(n):
        if layer is None:
            return rng.uniform(0, 0.5, n)
        i = np.arange(n)
        d = np.maximum(np.maximum(layer - i, i - (n - 1 - layer)), 0) / max(layer, 1)
        return 0.4 * d * d

    return wl.Workload(name=f"tile-{nx}x{ny}", nx=nx, ny=ny,
                       s=np.array([1.6, 1.6, 1.6, 1.1, 1.2, 1.3, 1.3, 1.9, 1.9]),
                       variant=variant, bc=bc, n=0.4, m=0.6, rho0=1.0, u0=(0.04, -0.02),
                       rho_f=1.002, u_f=(0.05, -0.01), chi_x=profile(nx), chi_y=profile(ny),
                       rho_dev=1e-3 * rng.standard_normal((ny, nx)), steps=7, storage="f32",
                       source=(1e-3, 0.07, 0.3) if bc == "channel" else (0.0, 0.0, 0.0))


def _state(w, storage, tiles, steps):
    from paper_1203_6350_gb300 import lbm

    with lbm.Lattice.from_workload(w, storage=storage) as lat:
        if not tiles:
            lat.steps_per_launch = 1  # names the launches
        for n in steps:
            launches = lbm.lbm_step_launches(lat.h, n)
            assert launches < n if tiles and n > 1 else launches == n
            lat.step(n)
        buf, t = lat.get_state()
        assert t == sum(steps)
        return buf


# a tile of 20 x 4 (up to 128^2 cells) or 24 x 16, one cell less and more, one cell
# rows and columns, lattices narrower than a region's halo, the largest of each class
@pytest.mark.parametrize("shape", [(2, 1), (1, 3), (3, 5), (19, 3), (20, 4), (21, 5), (127, 129),
                                   (4000, 4), (128, 129), (24, 700), (265, 191)])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic", "channel"])
@pytest.mark.parametrize("storage", ["f32", "f16dev", "bf16dev"])
def test_tiles_equal_a_launch_per_step(shape, bc, storage):
    nx, ny = shape
    if bc == "channel" and nx < 2:
        pytest.skip("a channel has two columns at least")
    for variant, layer in (("none", 0), ("I", 5), ("II", None), ("III", 5), ("viscous", 5)):
        if layer and 2 * layer >= min(nx, ny):
            layer = None
        w = _workload(nx, ny, bc, variant, layer, seed=nx * 31 + ny)
        steps = [2, 3, 1, 7, 130]  # single launches, replayed graphs and what they leave over
        a = _state(w, storage, True, steps)
        np.testing.assert_array_equal(a, _state(w, storage, False, steps), err_msg=variant)


def test_a_smaller_lattice_made_later_leaves_a_larger_one_its_tiles():
    """The kernels' shared-memory limit belongs to the process, not to a handle."""
    from paper_1203_6350_gb300 import lbm

    big, small = (_workload(n, n, "dirichlet", "II", 5, seed=n) for n in (200, 64))
    with lbm.Lattice.from_workload(big) as a, lbm.Lattice.from_workload(small) as b:
        b.step(12)
        a.step(12)
        got = a.get_state()[0]
    np.testing.assert_array_equal(got, _state(big, "f32", False, [12]))
