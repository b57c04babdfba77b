"""What a diverging iteration leaves behind: a batch ends with the system that diverges and solves again,
and the schedule tuner keeps nothing that it measured on updates that did no work."""
import ctypes

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


def _untuned(g):
    from paper_1611_06765_gb300 import _lib
    mask = ctypes.c_int()
    _lib.load().pnm_get_tuning(g._h, None, None, None, ctypes.byref(mask))
    return mask.value & 4


def test_diverging_updates_are_not_timed(pkg):
    """An interaction so strong that the residual overflows in the first update: the updates after it leave
    at once.  A solve that holds NaN tunes from the MBPT2 start."""
    strong = tuple(1e200 * v if k in (0, 2, 4) else v for k, v in enumerate(pkg.MINNESOTA))
    g = pkg.Context(14, 0.08, 5, params=strong)
    assert g.solve(alpha=0.5, tol=1e-8, max_iter=20, allow=(pkg.PNM_EDIVERGED,))[3] == pkg.PNM_EDIVERGED
    assert _untuned(g)
    g.close()
    g = pkg.Context(14, 0.08, 5)
    held = np.full(len(g.amplitude_labels()), np.nan)
    g.set_amplitudes(held)
    kw = dict(alpha=0.5, tol=1e-8, max_iter=60)
    assert g.solve(init=pkg.PNM_INIT_KEEP, allow=(pkg.PNM_EDIVERGED,), **kw)[3] == pkg.PNM_EDIVERGED
    assert not _untuned(g)
    assert g.solve(**kw)[3] == 0
    g.close()
