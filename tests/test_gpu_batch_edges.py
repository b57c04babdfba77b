"""End of an update over batches on both sides of the line where it takes one warp per system
instead of the whole block: the same updates and energies as each system alone."""
import numpy as np
import pytest

from conftest import minnesota_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_1611_06765_gb300 import build
    build.build()
    import paper_1611_06765_gb300 as P
    return P


@pytest.mark.parametrize("nsys", [1, 3, 4, 5, 9])
def test_batch_energies_equal_single_systems(pkg, nsys):
    """The energy of an update is a sum of FP64 partials in another order: 740 amplitudes per
    system bound the relative difference per update by 740 * 2^-53 < 1e-13 of the sum of
    absolute values, and the iteration only averages it; 1e-12 over the history."""
    P = minnesota_params()
    rhos = [0.04 + 0.02 * k for k in range(nsys)]
    kw = dict(alpha=0.5, tol=1e-8, max_iter=200)
    g = pkg.Context(14, rhos, 4, params=P)
    dE, it, _, _ = g.solve(**kw)
    for k, rho in enumerate(rhos):
        one = pkg.Context(14, rho, 4, params=P)
        dE1, it1, _, _ = one.solve(**kw)
        assert it1[0] == it[k]
        assert abs(dE1[0] - dE[k]) <= 1e-12 * abs(dE1[0])
        h, h1 = g.history(k), one.history(0)
        assert np.all(np.abs(h - h1) <= 1e-12 * np.abs(h1))
        one.close()
    g.close()
