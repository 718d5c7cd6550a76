"""FP16 storage where its scale S is large: a small porosity makes small deviations,
and S rho / eps would leave FP32's range.  Several steps per launch: tiles of
whole vectors and of odd rows, pairs."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_1601_00704_gb300 import build
    build.build()
    import paper_1601_00704_gb300 as p
    return p


# where the first scale (at most 2^64) leaves eps G S a normal FP16 number, the multi-step kernels are compared with single
# steps, within the rounding of a scale that may change at a chunk's end; beyond that the first chunk's length decides what
# is left of the deviations, and the velocity has to stay finite
@pytest.mark.parametrize("eps,G", [(1e-10, 1e-16), (1e-14, 1e-17), (1e-6, 1e-20), (1e-3, 1e-14), (0.1, 1e-6)])
@pytest.mark.parametrize("F_eps", [0.0, 0.7])
@pytest.mark.parametrize("nx,ny", [(64, 64), (67, 33), (1160, 1131)])
def test_small_porosity(pkg, nx, ny, F_eps, eps, G):
    n, u = 40, []
    for check in (1, 20):
        s = pkg.Solver(nx, ny, tau=0.8, storage="f16")
        s.set_medium(np.full((ny, nx), eps), np.full((ny, nx), eps), F_eps=F_eps)
        s.set_force(G)
        before = s.counters()[1]
        s.step(n, check_every=check)
        if check > 1:
            assert s.counters()[1] - before < n  # several steps per launch
        u.append(s.mean_velocity())
        assert np.isfinite(s.distributions()).all()
        s.close()
    assert np.isfinite(u).all()
    if eps * G * 2.0 ** 64 > 2.0 ** -14:
        assert abs(u[0][0] - u[1][0]) <= n * 2.0 ** -11 * abs(u[0][0])
