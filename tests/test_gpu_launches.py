"""lbm_step_launches against the step kernels that the device ran."""
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


def _kernels(work):
    """Names of the kernels that work() runs."""
    import torch
    from torch.profiler import ProfilerActivity, profile

    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        work()
        torch.cuda.synchronize()
    return [e.name for e in p.events()]


# tiles of six and of four levels, the channel over more than one source table, a lattice
# without tiles, a marching one
@pytest.mark.parametrize("shape,bc", [((100, 80), "channel"), ((210, 200), "channel"),
                                      ((300, 300), "channel"), ((100, 100), "periodic"),
                                      ((300, 200), "dirichlet"), ((1020, 803), "dirichlet")])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_the_launches_are_counted(shape, bc, mode):
    from paper_1203_6350_gb300 import lbm

    nx, ny = shape
    with lbm.Lattice(nx, ny, "f32", 1.0, (0.0, 0.0), 1.9, bc=bc) as lat:
        lbm.lbm_set_launch_mode(lat.h, mode)
        lat.init_pulse(1e-3, 5.0, nx / 2, ny / 2)
        lat.step(70)  # (graphs are built outside the count)
        for _ in range(2):  # (the first trace of a process may hold nothing)
            names = _kernels(lambda: lat.step(1))
        if not any("step" in n for n in names):
            pytest.skip("the profiler records no kernels here")
        for steps in (5, 64, 130, 192):
            names = _kernels(lambda: lat.step(steps))
            ran = sum("step2_kernel" in n or "tile_kernel" in n or "march_kernel" in n for n in names)
            assert ran == lbm.lbm_step_launches(lat.h, steps), (steps, set(names))
        assert np.isfinite(lat.moments()[0]).all()
