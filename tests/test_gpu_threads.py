"""Host threads with a handle or a stream each, at sizes whose kernels take
different amounts of shared memory: none is refused a launch because of another
(the limit of a kernel function is one for the whole process), and each gets
the results it gets alone."""

import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _together(jobs):
    """Run the jobs at the same time, several times each -> their results or exceptions."""
    out = [None] * len(jobs)
    start = threading.Barrier(len(jobs))

    def run(i):
        try:
            start.wait(60)
            out[i] = jobs[i]()
        except Exception as e:  # a refusal in a thread fails the test below
            out[i] = e

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(300)
    return out


@pytest.fixture(scope="module")
def pkg():
    from paper_1601_00704_gb300 import build
    build.build()
    import paper_1601_00704_gb300 as p
    p.load()
    return p


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_solvers_of_different_tiles(pkg, storage):
    import torch

    def job(nx, ny):
        stream = torch.cuda.Stream()

        def solve():
            s = pkg.Solver(nx, ny, storage=storage, stream=stream)
            eps = np.random.default_rng(nx).uniform(0.1, 0.2, (ny, nx))
            s.set_medium(eps, np.full((ny, nx), 1e-3))
            s.set_force(1e-6)
            s.step(6000, check_every=3)  # launched one by one
            for n in range(4, 40):       # a capture each
                s.step(n, check_every=n)
            f = s.distributions()
            s.close()
            return f
        return solve

    jobs = [job(512, 384), job(600, 260), job(128, 40)]
    alone = [j() for j in jobs]
    for a, b in zip(alone, _together(jobs)):
        assert isinstance(b, np.ndarray), b
        assert np.array_equal(a, b)
