"""Launches of several time steps on a user stream: captured chunks replayed from
either buffer and at step counts other than zero, with programmatic launches
and, in 16-bit storage, rounding keys from the device's step counter.  A state
that has settled (so that FP16 keeps its scale) goes through a checkpoint to
two solvers; one takes long chunks, the other single steps: the same bits."""

import pytest

import media

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_1601_00704_gb300 import build
    build.build()
    import paper_1601_00704_gb300 as p
    return p


# two steps a launch; tiles of whole vectors; tiles of odd rows (16-bit storage rounds node by node there)
CASES = [(480, 6000, st, F, w) for st in ("f32", "bf16", "f16") for F, w in ((0.0, True), (0.7, False))]
CASES += [(500, 200, st, F, w) for st in ("f32", "bf16", "f16") for F, w in ((0.0, True), (0.7, False))]
CASES += [(333, 70, st, 0.0, w) for st in ("f32", "bf16", "f16") for w in (True, False)]


@pytest.mark.parametrize("nx,ny,storage,F_eps,walls", CASES)
def test_replayed_chunks_are_the_single_steps(pkg, tmp_path, nx, ny, storage, F_eps, walls):
    import torch
    stream = torch.cuda.Stream()

    def solver():
        return pkg.Solver(nx, ny, tau=0.8, storage=storage, walls=walls, stream=stream)

    s = solver()
    s.set_medium(*media.random_medium(nx, ny, seed=nx), F_eps=F_eps)
    s.set_force(1e-5, 2e-6)
    s.step(300)
    path = str(tmp_path / "state")
    s.save(path)
    s.close()
    out = []
    for single in (False, True):
        s = solver()
        s.load(path)
        before = s.counters()[1]
        if single:
            s.step(149, check_every=1)
        else:
            s.step(70, check_every=17)   # chunks that start from either buffer, replayed
            s.step(79, check_every=16)
            assert s.counters()[1] - before < 115  # 149 steps; 10 finalizes and counter updates at most each
        fields = [torch.empty((9, ny, nx), dtype=torch.float64, device="cuda"),
                  torch.empty((ny, nx), dtype=torch.float64, device="cuda"),
                  torch.empty((ny, nx), dtype=torch.float64, device="cuda")]
        s.distributions(fields[0])
        s.velocity(*fields[1:])
        stream.synchronize()
        out.append(fields + [torch.from_numpy(s.mean_velocity())])
        assert s.guard_damage() == 0
        s.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
