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
          ((1024, 1024), "dirichlet", "f32", "II", 64, True),
          ((1024, 1024), "dirichlet", "f32", "II", 128, False),
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


V5 = ["none", "I", "II", "III", "viscous"]


# (instances as (count, shape), storage, variants in turn, marching)
@pytest.mark.parametrize("shapes,storage,variants,marching", [
    ([(4, (400, 390))], "f32", ["II"], True), ([(1, (700, 690))], "f32", ["I"], True),
    ([(16, (256, 250))], "f32", V5, True),
    ([(25, (64, 64)), (1, (1024, 1000))], "f32", ["II"], True),
    ([(4, (256, 256))], "f32", ["II"], False), ([(8, (190, 190))], "f32", ["III"], False),
    ([(32, (64, 1000))], "f32", ["II"], False), ([(64, (100, 100))], "f32", ["I"], False),
    ([(16, (256, 250))], "f16dev", ["II"], True), ([(2, (160, 170))], "bf16dev", ["II"], True),
    ([(40, (200, 190))], "bf16dev", V5, True),
    ([(30, (64, 64)), (1, (2048, 1500))], "f16dev", ["none"], True),
    ([(32, (64, 1000))], "f16dev", ["III"], False), ([(30, (200, 200))], "bf16dev", ["I"], False),
    ([(16, (128, 130))], "f16dev", ["II"], False)])
def test_batches_march_where_it_is_faster(shapes, storage, variants, marching, monkeypatch):
    from test_gpu_launches import _kernels

    from paper_1203_6350_gb300.batch import Batch

    def fields(expect):
        with Batch(storage, config={"cells": 2, "steps_per_launch": 2, "tile": (64, 16)}) as b:
            ids = []
            for count, (nx, ny) in shapes:
                for _ in range(count):
                    v = variants[len(ids) % len(variants)]
                    w = 0 if v == "none" else 20
                    i = b.add(nx, ny, 1000, s=1.6, u0=(0.04, -0.02), variant=v,
                              chi_x=_ramp(nx, w), chi_y=_ramp(ny, w))
                    b.init_pulse(i, 1e-3, 6.0, 0.4 * nx, 0.6 * ny)
                    ids.append(i)
            b.step(1)
            for _ in range(2):  # (the first trace of a process may hold nothing)
                names = _kernels(lambda: b.step(12))
            if any("batch" in n for n in names):
                assert any("march_batch" in n for n in names) == expect
            for n in (4, 7, 35):
                b.step(n)
            return [b.moments(i) for i in ids]

    monkeypatch.delenv("LBM_BATCH_TMA", raising=False)
    got = fields(marching)
    monkeypatch.setenv("LBM_BATCH_TMA", "1")
    for a, b in zip(got, fields(False)):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("storage,steps", [("f32", 4), ("f32", 8), ("f16dev", 5)])
def test_a_short_call_moves_the_clock_once(storage, steps):
    """The steps that marching launches leave over read the clock at an offset."""
    from test_gpu_launches import _kernels

    from paper_1203_6350_gb300.batch import Batch

    with Batch(storage, config={"cells": 2, "steps_per_launch": 2, "tile": (64, 16)}) as b:
        i = b.add(700, 690, 1000, s=1.6)
        b.init_pulse(i, 1e-3, 6.0, 300.0, 300.0)
        b.step(1)
        for _ in range(2):  # (the first trace of a process may hold nothing)
            names = _kernels(lambda: b.step(steps))
        if any("batch" in n for n in names):
            assert any("march_batch" in n for n in names)
            assert sum("advance_counters" in n for n in names) == 1
        assert b.time(i) == 1 + 2 * steps
