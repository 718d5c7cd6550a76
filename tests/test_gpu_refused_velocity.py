"""The velocity field after a refused step call (glbm_debug_fail_launch refuses a
launch on the host; nothing faults) is that of the last step that ran, also
where a launch advances several steps: bit for bit that of a solver that takes
the same steps one by one."""

import numpy as np
import pytest

import media

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    from paper_1601_00704_gb300 import build
    build.build()
    import torch

    import paper_1601_00704_gb300 as pkg
    lib = pkg.load()
    yield pkg, lib, torch
    lib.glbm_debug_fail_launch(-1)


def _solver(pkg, nx, ny, storage, stream=None, F_eps=0.0):
    s = pkg.Solver(nx, ny, tau=0.8, storage=storage, stream=stream)
    s.set_medium(*media.random_medium(nx, ny, seed=nx), F_eps=F_eps)
    s.set_force(1e-4, 2e-5)
    return s


# tiles of several steps (whole vectors and odd rows), pairs of steps, one step a launch (f64)
SHAPES = [(128, 96, "f32"), (128, 96, "bf16"), (333, 70, "f32"), (1160, 1131, "f32"), (128, 96, "f64")]


@pytest.mark.parametrize("nx,ny,storage", SHAPES)
@pytest.mark.parametrize("after", [0, 6, 14])
def test_refusal_in_a_chunk_launched_directly(env, nx, ny, storage, after):
    pkg, lib, torch = env
    s = _solver(pkg, nx, ny, storage)
    s.step(10, check_every=5)
    lib.glbm_debug_fail_launch(after)
    try:
        with pytest.raises(pkg.GLBMError):
            s.step(40, check_every=40)
    finally:
        lib.glbm_debug_fail_launch(-1)
    f, u = s.distributions(), s.velocity()
    ref = _solver(pkg, nx, ny, storage)
    ref.step(10, check_every=1)
    while not np.array_equal(ref.distributions(), f):
        assert ref.counters()[0] <= 10 + after
        ref.step(1, check_every=1)
    assert all(np.array_equal(a, b) for a, b in zip(ref.velocity(), u))
    assert np.array_equal(s.distributions(), f)
    s.step(12, check_every=1)
    ref.step(12, check_every=1)
    assert np.array_equal(s.distributions(), ref.distributions())


@pytest.mark.parametrize("nx,ny,storage", SHAPES)
@pytest.mark.parametrize("chunk", [60, 63])
def test_refusal_while_a_later_chunk_is_captured(env, nx, ny, storage, chunk):
    pkg, lib, torch = env
    s = _solver(pkg, nx, ny, storage, stream=torch.cuda.Stream(), F_eps=0.7)
    lib.glbm_debug_fail_launch(chunk + 5)  # the first chunk is captured; refused in the next capture
    try:
        with pytest.raises(pkg.GLBMError):
            s.step(2 * chunk + 10, check_every=chunk)
    finally:
        lib.glbm_debug_fail_launch(-1)
    done = s.counters()[0]
    assert done in (chunk, 2 * chunk)  # the second chunk is replayed, unless it starts from the other buffer
    u = s.velocity()
    ref = _solver(pkg, nx, ny, storage, F_eps=0.7)
    ref.step(done, check_every=1)
    assert np.array_equal(ref.distributions(), s.distributions())
    assert all(np.array_equal(a, b) for a, b in zip(ref.velocity(), u))
