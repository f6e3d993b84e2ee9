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


# the tiles of 4 and of 16 rows that the device holds at once, and one more (152 SMs): steps of
# a launch
@pytest.mark.parametrize("shape,levels", [((3040, 5), 6), ((3041, 5), 4), ((1824, 25), 4),
                                          ((1825, 25), 1), ((1, 1216), 6), ((1, 1217), 4),
                                          ((1, 2433), 1), ((17000, 3), 1), ((16000, 1), 1)])
@pytest.mark.parametrize("storage", ["f32", "f16dev", "bf16dev"])
def test_tiles_only_where_they_fit_the_device_at_once(shape, levels, storage):
    import torch
    from paper_1203_6350_gb300 import lbm

    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the shapes are those of 152 SMs")
    with lbm.Lattice(*shape, storage, 1.0, (0.0, 0.0), 1.9) as lat:
        assert lbm.lbm_step_launches(lat.h, 12) == 12 // levels
        lat.init_pulse(1e-3, 5.0, shape[0] / 2, shape[1] / 2)
        lat.step(13)
        got, _ = lat.get_state()
    with lbm.Lattice(*shape, storage, 1.0, (0.0, 0.0), 1.9) as lat:
        lat.steps_per_launch = 1
        lat.init_pulse(1e-3, 5.0, shape[0] / 2, shape[1] / 2)
        lat.step(13)
        np.testing.assert_array_equal(got, lat.get_state()[0])
