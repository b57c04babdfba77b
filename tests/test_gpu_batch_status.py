"""How a batch of systems ends: one that diverges ends the solve of all, and leaves nothing behind."""
import numpy as np
import pytest

from inputs import random_amplitudes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_1611_06765_gb300 import build
    build.build()
    import paper_1611_06765_gb300 as P
    return P


@pytest.mark.parametrize("nsys", [1, 2, 7])
@pytest.mark.parametrize("mixed", [False, True])
def test_one_system_diverges(pkg, nsys, mixed):
    g = pkg.Context(14, [0.08 + 0.01 * k for k in range(nsys)], 4)
    kw = dict(alpha=0.5, tol=1e-8, max_iter=60)
    if mixed:
        kw.update(precision=pkg.PNM_PREC_BF16X3, refine_sweeps=2)
    first = g.solve(**kw)
    assert first[3] == 0
    held = [g.get_amplitudes(k) for k in range(nsys)]
    bad = random_amplitudes(len(held[nsys // 2]), seed=2)
    bad[5] = np.nan
    g.set_amplitudes(bad, sys=nsys // 2)
    rc = g.solve(init=pkg.PNM_INIT_KEEP, allow=(pkg.PNM_EDIVERGED,), **kw)[3]
    assert rc == pkg.PNM_EDIVERGED
    again = g.solve(**kw)
    assert again[3] == 0 and np.array_equal(again[0], first[0]) and np.array_equal(again[1], first[1])
    for k in range(nsys):
        assert np.array_equal(g.get_amplitudes(k), held[k])
    g.close()
