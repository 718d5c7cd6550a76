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


# (kernel, two layers of it: n, h, w, input channels, output channels) that take different amounts of shared memory
LAYERS = {"streaming": ((1, 600, 256, 32, 64), (1, 600, 256, 64, 64)), "band": ((1, 16, 256, 32, 64), (1, 16, 256, 64, 64)),
          "tile": ((2, 40, 40, 32, 256), (2, 40, 40, 32, 96)), "weight gradient": ((2, 16, 16, 32, 32), (2, 64, 64, 64, 64))}


@pytest.mark.parametrize("kernel", LAYERS)
def test_layers_of_different_sizes(pkg, kernel):
    import ctypes as C

    import torch
    lib = pkg.load()

    def vp(t):
        return C.c_void_p(t.data_ptr())

    def job(n, h, w, ci, co):
        g = torch.Generator(device="cuda").manual_seed(ci + co)
        x = torch.randn((n, h, w, ci), generator=g, device="cuda").to(torch.bfloat16)
        dy = torch.randn((n, h, w, co), generator=g, device="cuda").to(torch.bfloat16)
        wt = torch.randn((9, co, ci), generator=g, device="cuda").to(torch.bfloat16)
        b = torch.randn(co, generator=g, device="cuda")
        y = torch.empty((n, h, w, co), dtype=torch.bfloat16, device="cuda")
        dw = torch.zeros((co, ci, 3, 3), device="cuda")
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        stream = torch.cuda.Stream()
        st = C.c_void_p(stream.cuda_stream)
        torch.cuda.synchronize()

        def layer():
            torch.cuda.set_device(0)  # the thread's CUDA context, which encoding a tensor map needs
            torch.cuda.synchronize()
            for _ in range(1500):
                if kernel == "weight gradient":
                    rc = lib.glbm_nn_tc_conv_wgrad(vp(x), ci, ci, vp(dy), co, co, n, h, w, 3, vp(dw), vp(err), st)
                else:
                    rc = lib.glbm_nn_tc_conv(vp(x), ci, None, 0, n, h, w, 3, vp(wt), vp(b), co, vp(y), co, 1, 0, 0,
                                             vp(err), st)
                if rc != 0:
                    raise pkg.GLBMError(rc, lib.glbm_last_error(None).decode())
            stream.synchronize()
            assert int(err) == 0
            return y.clone()
        return layer

    jobs = [job(*shape) for shape in LAYERS[kernel]]
    alone = [j() for j in jobs]
    for a, b in zip(alone, _together(jobs)):
        assert isinstance(b, torch.Tensor), b
        assert kernel == "weight gradient" or torch.equal(a, b)
