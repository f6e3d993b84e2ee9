"""Steps captured into a graph of the caller's: each replay goes on from where the last
one ended, as it does with the launches that the handle's settings name."""
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


def _workload(nx, ny, bc, seed):
    rng = np.random.default_rng(seed)
    chi = [np.where((np.arange(n) < 6) | (np.arange(n) >= n - 6), 0.2, 0.0) for n in (nx, ny)]
    return wl.Workload(name=f"capture-{nx}x{ny}", nx=nx, ny=ny, s=np.full(9, 1.7), variant="II",
                       bc=bc, n=0.4, m=0.6, rho0=1.0, u0=(0.04, -0.02), rho_f=1.0,
                       u_f=(0.04, -0.02), chi_x=chi[0], chi_y=chi[1],
                       rho_dev=1e-3 * rng.standard_normal((ny, nx)), steps=1, storage="f32",
                       source=(1e-3, 0.07, 0.3) if bc == "channel" else (0.0, 0.0, 0.0))


def _graph(stream, work):
    import torch

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        work()
    return g


# tiles of six and of four levels, their channel over more than one source table, marching
# lattices with one and with two steps to a named launch
@pytest.mark.parametrize("shape,bc,steps", [
    ((100, 100), "dirichlet", 2), ((100, 100), "dirichlet", 6), ((100, 100), "periodic", 64),
    ((100, 80), "channel", 130), ((200, 200), "dirichlet", 6), ((210, 200), "channel", 100),
    ((1020, 803), "dirichlet", 14), ((1501, 1405), "dirichlet", 8),
    ((1501, 1405), "dirichlet", 20), ((1504, 1405), "periodic", 32)])
@pytest.mark.parametrize("storage", ["f32", "f16dev", "bf16dev"])
def test_replays_of_captured_steps_go_on(shape, bc, steps, storage):
    import torch
    from paper_1203_6350_gb300 import lbm

    w = _workload(*shape, bc, seed=sum(shape))
    stream = torch.cuda.Stream()
    with lbm.Lattice.from_workload(w, storage=storage, stream=stream) as lat:
        lat.step(2 * steps)
        graph = _graph(stream, lambda: lat.step(steps))
        with torch.cuda.stream(stream):
            for _ in range(3):
                graph.replay()
        got, _ = lat.get_state()
    with lbm.Lattice.from_workload(w, storage=storage) as lat:
        lat.steps_per_launch = lat.steps_per_launch
        lat.step(2 * steps)
        for _ in range(3):
            lat.step(steps)
        want, _ = lat.get_state()
    np.testing.assert_array_equal(got, want)


def test_a_batch_steps_on_after_replays(monkeypatch):
    """Replays advance the device's step counter alone, and a budget ends by that counter."""
    import torch
    from paper_1203_6350_gb300.batch import Batch

    works = [_workload(420, 400, "dirichlet", seed=1), _workload(430, 390, "dirichlet", seed=2)]
    budgets = [20, 1000]
    config = {"cells": 2, "steps_per_launch": 2, "tile": (64, 16)}

    def fields(replays):
        stream = torch.cuda.Stream()
        with Batch("f32", stream=stream, config=config) as b:
            ids = [b.add_workload(w, steps=n) for w, n in zip(works, budgets)]
            b.step(4)
            if replays:  # 4 steps, then 3 x 4 replayed, then 12 more
                graph = _graph(stream, lambda: b.step(4))
                with torch.cuda.stream(stream):
                    for _ in range(3):
                        graph.replay()
                b.step(12)
            else:
                b.step(24)
            return [b.moments(i) for i in ids]

    monkeypatch.delenv("LBM_BATCH_TMA", raising=False)
    got = fields(True)
    monkeypatch.setenv("LBM_BATCH_TMA", "1")  # the tile kernels throughout
    for a, b in zip(got, fields(False)):
        np.testing.assert_array_equal(a, b)
