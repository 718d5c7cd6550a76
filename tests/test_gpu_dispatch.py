"""Lattices near the lines between one step, two steps and several steps per launch:
the kernels on the slower side of a line are not taken (launches of a chunk are
counted), and whichever is taken gives the bits of single steps."""

import numpy as np
import pytest

import media

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_1601_00704_gb300 import build
    build.build()
    import paper_1601_00704_gb300 as p
    return p


# (nx, ny, storage, F_eps, time steps per launch).  Measured, us a step, one step per launch / several: 1000 x 500 BF16 3.95 / 4.54, 1021 x 587 FP32 7.0 / 10.2 and BF16 8.8 / 11.7, 1021 x 391 FP32 with
# Forchheimer 5.1 / 6.2, 1024 x 1367 BF16 8.6 / 10.9; 1000 x 240 BF16 2.88 / 2.31, 100 x 3000 FP32 8.4 / 3.5,
# 128 x 10937 BF16 27 / 15, 1024 x 1367 FP32 13.3 / 10.3 (Forchheimer 14.3 / 11.6)
LINES = [(1000, 500, "bf16", 0.0, 1), (1021, 587, "bf16", 0.0, 1), (1021, 391, "f32", 0.7, 1), (1024, 1367, "bf16", 0.0, 1),
         (1024, 1367, "bf16", 0.7, 1), (1000, 240, "bf16", 0.0, 4), (100, 3000, "f32", 0.0, 4), (128, 10937, "bf16", 0.0, 2),
         (1024, 1367, "f32", 0.0, 2), (1024, 1367, "f32", 0.7, 2)]


@pytest.mark.parametrize("nx,ny,storage,F_eps,per_launch", LINES)
def test_steps_per_launch(pkg, nx, ny, storage, F_eps, per_launch):
    import torch
    medium = [torch.from_numpy(a).cuda() for a in media.random_medium(nx, ny, seed=nx)]
    out = []
    for check in (41, 1):
        stream = torch.cuda.Stream()
        s = pkg.Solver(nx, ny, tau=0.8, storage=storage, stream=stream)
        torch.cuda.synchronize()
        s.set_medium(*medium, F_eps=F_eps)
        s.set_force(1e-4, 2e-5)
        before = s.counters()[1]
        s.step(41, check_every=check)
        launched = s.counters()[1] - before
        if check == 41:  # 40 steps, the reducing one, its finalize and in 16-bit storage the step counter
            assert launched == 40 // per_launch + 2 + (storage != "f32")
        f = torch.empty((9, ny, nx), dtype=torch.float64, device="cuda")
        s.distributions(f)
        stream.synchronize()
        out.append(f)
        s.close()
    assert torch.equal(*out)


def test_plan_follows_the_medium(pkg):
    """The same handle with and without Forchheimer drag: another kernel from the new medium's first chunk on."""
    import torch
    nx, ny = 1021, 391
    stream = torch.cuda.Stream()
    s = pkg.Solver(nx, ny, stream=stream)
    medium = media.random_medium(nx, ny, seed=1)
    counts = []
    for F_eps in (0.0, 0.7, 0.0):
        s.set_medium(*medium, F_eps=F_eps)
        s.set_force(1e-4)
        before = s.counters()[1]
        s.step(41, check_every=41)
        counts.append(s.counters()[1] - before)
        f = s.distributions()
        r = pkg.Solver(nx, ny)
        r.set_medium(*medium, F_eps=F_eps)
        r.set_force(1e-4)
        r.step(41, check_every=1)
        assert np.array_equal(f, r.distributions())
        r.close()
    assert counts[1] == 42 and counts[0] == counts[2] < 20
