"""The batched marching launches (the default for two-step batches of larger Dirichlet
instances) against the batched tile kernels: the fields agree bit for bit."""
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


def _fields(works, budgets, storage, calls):
    from paper_1203_6350_gb300.batch import Batch

    with Batch(storage, config={"cells": 2, "steps_per_launch": 2, "tile": (64, 16)}) as b:
        ids = []
        for k, (w, n) in enumerate(zip(works, budgets)):
            ids.append(b.add_workload(w, steps=n, init="pulse"))
            if k % 5 == 2:
                b.step(1 + k % 4)  # later instances start at later steps
        for n in calls:
            b.step(n)
        return [b.moments(i) for i in ids], [b.time(i) for i in ids]


# 40 instances of one variant need two launches; budgets end inside a launch's steps
@pytest.mark.parametrize("case", ["mixed", "one variant", "none and viscous"])
@pytest.mark.parametrize("storage", ["f32", "f16dev", "bf16dev"])
def test_marching_batches_equal_the_tiles(case, storage, monkeypatch):
    works = wl.batch_of_lattices(seed=5, count=40 if case == "one variant" else 13, lo=130, hi=420,
                                 storage=storage)
    if case == "one variant":
        works = [w.with_(variant="II") for w in works]
    elif case == "none and viscous":
        works = [w.with_(variant="none" if k % 2 else "viscous",
                         chi_x=wl.viscous_ramp(w.nx, w.width), chi_y=wl.viscous_ramp(w.ny, w.width))
                 for k, w in enumerate(works)]
    budgets = [23 + 7 * (k % 6) for k in range(len(works))]
    monkeypatch.delenv("LBM_BATCH_TMA", raising=False)
    got, t = _fields(works, budgets, storage, [1, 2, 9, 40])
    monkeypatch.setenv("LBM_BATCH_TMA", "1")
    want, u = _fields(works, budgets, storage, [1, 2, 9, 40])
    assert t == u
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)
