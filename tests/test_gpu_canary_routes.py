"""Padding canaries under the kernels that a handle or batch takes by default: marching, tiles
of several steps, batched marching.  The padding keeps its all-one bytes and no NaN of it
reaches a cell (test_gpu_canary.py has the kernels that are asked for by name)."""
import numpy as np
import pytest

from test_gpu_canary import ES, _split

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6350_gb300 import lbm

    lbm.load()


def _ramp(n, width):
    i = np.arange(n)
    d = np.clip(width - np.minimum(i, n - 1 - i), 0, width) / max(width, 1)
    return 0.3 * d * d


def _canary(monkeypatch, on):
    if on:
        monkeypatch.setenv("LBM_CANARY", "1")
    else:
        monkeypatch.delenv("LBM_CANARY", raising=False)


def _fields(shape, seed):
    rng = np.random.default_rng(seed)
    nx, ny = shape
    return (1.0 + 1e-3 * rng.standard_normal((ny, nx)), np.full((ny, nx), 0.04),
            np.full((ny, nx), -0.02))


def _check(with_canary, without, rows, nx, storage):
    cells_c, pad = _split(with_canary, rows, nx, ES[storage])
    cells, _ = _split(without, rows, nx, ES[storage])
    assert pad.size > 0 and np.all(pad == 0xFF), "a kernel wrote into the row padding"
    np.testing.assert_array_equal(cells_c, cells)


# rows that end 1 to 3 elements into a staged chunk, in the last strip or just past it
CASES = [(s, "dirichlet", 20) for s in ((1019, 811), (901, 899), (1022, 787), (2051, 1999))] + [
    ((1401, 1405), "periodic", 20), ((1204, 1001), "periodic", 20)] + [
    (s, bc, 2) for s in ((21, 5), (127, 129), (265, 191)) for bc in ("dirichlet", "periodic", "channel")]


@pytest.mark.parametrize("shape,bc,width", CASES)
@pytest.mark.parametrize("storage", ["f32", "f16dev", "bf16dev"])
def test_the_default_kernels_leave_padding_alone(monkeypatch, shape, bc, width, storage):
    from paper_1203_6350_gb300 import lbm

    nx, ny = shape
    if bc == "periodic" and nx == 1401 and storage != "f32":
        pytest.skip("16-bit periodic rows that are no multiple of 4 do not march")
    for variant in ("none", "II"):
        states = []
        for canary in (True, False):
            _canary(monkeypatch, canary)
            with lbm.Lattice(nx, ny, storage, 1.0, (0.04, -0.02), 1.6, bc=bc) as lat:
                lat.set_sponge(variant, _ramp(nx, width), _ramp(ny, width))
                lat.init_equilibrium(*_fields(shape, seed=nx))
                launches = lbm.lbm_step_launches(lat.h, 12)
                assert launches < 12 // lat.steps_per_launch or (
                    launches == 6 and storage != "f32")  # 16-bit above L2: two steps in either way
                lat.step(13)
                states.append(lat.get_state()[0])
        _check(*states, 9 * ny, nx, storage)


@pytest.mark.parametrize("storage", ["f32", "f16dev", "bf16dev"])
def test_batched_marching_leaves_padding_alone(monkeypatch, storage):
    from test_gpu_launches import _kernels

    from paper_1203_6350_gb300.batch import Batch

    shapes = [(451, 389), (517, 413), (389, 521), (601, 403), (481, 419)]
    states = []
    for canary in (True, False):
        _canary(monkeypatch, canary)
        with Batch(storage, config={"cells": 2, "steps_per_launch": 2, "tile": (64, 16)}) as b:
            ids = []
            for k, s in enumerate(shapes):
                w = 0 if k == 0 else 20
                i = b.add(*s, 30, s=1.6, u0=(0.04, -0.02), chi_x=_ramp(s[0], w),
                          chi_y=_ramp(s[1], w), variant=("none", "I", "II", "III", "viscous")[k])
                b.init_equilibrium(i, *_fields(s, seed=k))
                ids.append(i)
            for _ in range(2):
                names = _kernels(lambda: b.step(12))
            if any("batch" in n for n in names):
                assert any("march_batch" in n for n in names)
            b.step(20)
            states.append([b.get_state(i) for i in ids])
    for s, a, c in zip(shapes, *states):
        _check(a, c, 9 * s[1], s[0], storage)
