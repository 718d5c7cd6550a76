"""The one-launch EM iteration at the edges of its blocks (256 samples, 304
blocks), for every number of components, and where its variance update would
cancel and the two-pass iteration takes over.  Against the FP64 oracle: sums
in another order, so 1e-9 relative as in test_gpu_em.py."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_1601_00704_gb300 import build
    build.build()
    import paper_1601_00704_gb300 as p
    return p


def check(pkg, orc, x, init, iters):
    for it in iters:
        a = pkg.em_gmm1d(x, *init, max_iter=it, tol=0.0)
        b = orc.em_gmm1d(x, *init, max_iter=it, tol=0.0)
        assert a[3] == b[3] == it
        for u, v in zip(a[:3], b[:3]):
            np.testing.assert_allclose(u, v, rtol=1e-9, atol=1e-12)
        assert a[4] == pytest.approx(b[4], rel=1e-12)


@pytest.mark.parametrize("m,k", [(127, 1), (128, 1), (129, 2), (255, 2), (256, 3), (257, 1), (1000, 8), (4096, 5), (77823, 2), (77824, 3),
                                 (77825, 4), (200001, 6), (130000, 7)])
def test_block_edges_and_components(pkg, orc, m, k):
    rng = np.random.default_rng(m + k)
    x = rng.normal(3.0 + 4.0 * rng.integers(0, k, m), 1.0 + 0.3 * rng.random(m))
    init = (np.full(k, 1.0 / k), np.linspace(2.5, 4.0 * k, k), np.full(k, 4.0))
    check(pkg, orc, x, init, (1, 2, 17))


@pytest.mark.parametrize("start", [-50.0, 12.0, 1e4])
def test_mean_far_from_the_samples(pkg, orc, start):
    """The first iteration moves the mean by many sigma: its one-pass variance
    would cancel, so the two-pass form runs; the next ones are one-pass."""
    rng = np.random.default_rng(1)
    x = rng.normal(7.0, 0.25, 5000)
    check(pkg, orc, x, ([1.0], [start], [1.0e6]), (1, 3))


def test_tolerance_stops_between_batches(pkg, orc):
    rng = np.random.default_rng(9)
    x = np.concatenate([rng.normal(10, 1.5, 3000), rng.normal(14, 2.0, 5000)])
    init = ([0.5, 0.5], [8.0, 18.0], [9.0, 9.0])
    for tol in (1e-2, 1e-4, 1e-6, 1e-8):
        a = pkg.em_gmm1d(x, *init, max_iter=300, tol=tol)
        b = orc.em_gmm1d(x, *init, max_iter=300, tol=tol)
        assert a[3] == b[3]
        np.testing.assert_allclose(a[1], b[1], rtol=1e-9)
