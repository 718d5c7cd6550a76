"""bench.py's count of the launches that are not step kernels, by which it
counts the bytes of a time step."""

import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_under_test", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


@pytest.mark.parametrize("storage,n,check,tested,other", [
    ("f32", 300, 100, False, 1), ("bf16", 300, 100, False, 4), ("f16", 300, 100, False, 6), ("f32", 2500, 1000, True, 3),
    ("bf16", 2500, 1000, True, 6), ("f64", 10, 100, False, 1)])
def test_other_launches(bench, storage, n, check, tested, other):
    assert bench.other_launches(n, storage, check, tested) == other


@pytest.mark.gpu
@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
def test_step_launches_of_a_large_lattice(bench, storage):
    """2048 x 2048: pairs of steps, and at the end of a chunk that reduces (FP16: each, else the last) two single ones."""
    import numpy as np
    import torch

    from paper_1601_00704_gb300 import build
    build.build()
    import paper_1601_00704_gb300 as pkg
    s = pkg.Solver(2048, 2048, storage=storage, stream=torch.cuda.Stream())
    s.set_medium(np.full((2048, 2048), 0.1), np.full((2048, 2048), 1e-3))
    s.set_force(1e-6)
    s.step(300)  # FP16 settles its scale
    l0 = s.counters()[1]
    s.step(300)
    assert s.counters()[1] - l0 - bench.other_launches(300, storage) == (153 if storage == "f16" else 151)
