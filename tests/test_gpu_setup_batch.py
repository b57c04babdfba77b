"""The setup kernels take every system of a context in one launch: a system's tables do not depend on
the others of its context, whatever their sizes, species and twists, and its errors are still found."""
import numpy as np
import pytest

import paper_1611_06765_gb300 as P

pytestmark = pytest.mark.gpu

# (N, Z, rho, n2max, theta): smallest and larger boxes side by side, protons, twists
SYSTEMS = [
    (2, 0, 0.05, 1, None),
    (14, 0, 0.08, 9, None),
    (14, 14, 0.16, 4, None),
    (14, 0, 0.08, 6, (0.7, 1.1, 0.3)),
    (66, 0, 0.16, 12, None),
    (0, 14, 0.12, 5, None),
]


def _context(systems):
    theta = [s[4] or (0.0, 0.0, 0.0) for s in systems]
    return P.Context([s[0] for s in systems], [s[2] for s in systems], [s[3] for s in systems],
                     Z=[s[1] for s in systems], theta=np.array(theta))


def _tables(ctx, k):
    n, eps, holes = ctx.basis(k)
    out = [n, eps, np.array([ctx.eref()[k], ctx.mbpt2()[k]]), ctx.amplitude_labels(k)]
    for kind in (0, 1):
        out += list(ctx.channels(k, kind))
    return [np.asarray(x) for x in out] + [np.asarray(holes)]


@pytest.mark.parametrize("order", [(0, 1, 2, 3, 4, 5), (4, 0, 5, 2), (3, 4, 1, 0)])
def test_systems_of_a_batch_equal_their_own_contexts(order):
    with _context([SYSTEMS[k] for k in order]) as ctx:
        for k, o in enumerate(order):
            with _context([SYSTEMS[o]]) as alone:
                # whole numbers and sums alike, bit for bit
                for a, b in zip(_tables(ctx, k), _tables(alone, 0)):
                    assert np.array_equal(a, b), o
                # the index maps and V blocks through the two operators: the kernels chosen for a
                # context may differ, each within a few hundred roundings of its sums
                t = np.random.default_rng(o).uniform(-1, 1, len(ctx.amplitude_labels(k)))
                for op in ("apply_pp_ladder", "apply_ph_term"):
                    a, b = getattr(ctx, op)(t, sys=k), getattr(alone, op)(t)
                    assert np.max(np.abs(a - b), initial=0.0) <= 1e-12 * max(1.0, np.max(np.abs(b), initial=0.0)), (o, op)


@pytest.mark.parametrize("bad", [(13, 0, 0.08, 9, None), (14, 0, 0.08, 1, None), (14, 7, 0.08, 9, None), (10, 0, 0.08, 9, (0.0, 0.0, 0.5))])
@pytest.mark.parametrize("place", [0, 1, 2])
def test_one_refused_system_refuses_the_batch(bad, place):
    systems = [SYSTEMS[1], SYSTEMS[4]]
    systems.insert(place, bad)
    with pytest.raises(P.PnmError):
        _context(systems)
