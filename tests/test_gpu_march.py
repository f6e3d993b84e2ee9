"""The marching kernels (several steps per launch, the default on large
lattices) against the one-step and two-step launches on the same lattices: the
stored states agree bit for bit."""
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
    """Random deviations; chi random everywhere (layer None), or a quadratic ramp
    `layer` cells deep around a chi = 0 core."""
    rng = np.random.default_rng(seed)

    def profile(n):
        if layer is None:
            return rng.uniform(0, 0.5, n)
        i = np.arange(n)
        d = np.maximum(np.maximum(layer - i, i - (n - 1 - layer)), 0) / max(layer, 1)
        return 0.4 * d * d

    return wl.Workload(name=f"march-{nx}x{ny}", nx=nx, ny=ny,
                       s=np.array([1.6, 1.6, 1.6, 1.1, 1.2, 1.3, 1.3, 1.9, 1.9]),
                       variant=variant, bc=bc, n=0.4, m=0.6, rho0=1.0, u0=(0.04, -0.02),
                       rho_f=1.002, u_f=(0.05, -0.01), chi_x=profile(nx), chi_y=profile(ny),
                       rho_dev=1e-3 * rng.standard_normal((ny, nx)), steps=7, storage="f32")


def _state(w, storage, march, steps):
    from paper_1203_6350_gb300 import lbm

    with lbm.Lattice.from_workload(w, storage=storage) as lat:
        if not march:
            lat.steps_per_launch = lat.steps_per_launch  # names the launches
        for n in steps:
            if march and storage == "f32":  # three steps a launch, and what is left over
                assert lbm.lbm_step_launches(lat.h, n) <= n // 3 + 2
            lat.step(n)
        buf, t = lat.get_state()
        assert t == sum(steps)
        return buf


# widths of 0, 1 and 59 columns past a strip of 60, odd rows, one that is just high
# enough, and 16-bit states above L2 (two steps per rounding)
SHAPES = [(1020, 803), (901, 899), (1019, 811), (240, 3401), (13001, 64), (2051, 1999)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("variant,layer", [("none", 0), ("I", 37), ("II", None), ("II", 20),
                                           ("III", 37), ("viscous", 29)])
@pytest.mark.parametrize("storage", ["f32", "f16dev", "bf16dev"])
def test_marching_equals_the_launches_it_replaces(shape, variant, layer, storage):
    w = _workload(*shape, "dirichlet", variant, layer, seed=shape[0] + shape[1])
    steps = [7, 70] if shape[0] < 1000 else [8]
    a = _state(w, storage, True, steps)
    np.testing.assert_array_equal(a, _state(w, storage, False, steps))


@pytest.mark.parametrize("shape", [(1200, 1001), (1401, 1405), (2052, 1999)])
@pytest.mark.parametrize("variant,layer", [("none", 0), ("I", 37), ("II", None), ("III", 20),
                                           ("viscous", 29)])
@pytest.mark.parametrize("storage", ["f32", "f16dev", "bf16dev"])
def test_periodic_marching_equals_the_launches_it_replaces(shape, variant, layer, storage):
    w = _workload(*shape, "periodic", variant, layer, seed=shape[0] + shape[1])
    a = _state(w, storage, True, [8])
    np.testing.assert_array_equal(a, _state(w, storage, False, [8]))
