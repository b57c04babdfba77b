"""The updates take chunks of 32 amplitudes, one to four per warp by the size of the context, and each
system is closed by its own last block: a system's iteration does not depend on the others of its context."""
import numpy as np
import pytest

import paper_1611_06765_gb300 as P

pytestmark = pytest.mark.gpu

CAP = dict(alpha=0.5, max_iter=4, tol=1e-30, allow=(P.PNM_ENOTCONV,))


# N = 14, n^2 <= 20 has about 430 chunks: one, two and four of them per warp from 46 and 91 systems on
@pytest.mark.parametrize("systems", [2, 50, 100])
@pytest.mark.parametrize("prec,rtol", [(P.PNM_PREC_FP64, 1e-12), (P.PNM_PREC_BF16X3, 1e-5)])
def test_chunks_per_warp(systems, prec, rtol):
    rho = np.linspace(0.05, 0.15, systems)
    with P.Context(14, rho, 20) as ctx:
        dE, it, res, _ = ctx.solve(precision=prec, **CAP)
        for k in (0, systems // 2, systems - 1):
            with P.Context(14, rho[k], 20) as alone:
                e1, i1, r1, _ = alone.solve(precision=prec, **CAP)
            # sums of the same terms in another order: FP64, or FP32 terms with other splits
            assert it[k] == i1[0]
            assert abs(dE[k] - e1[0]) <= rtol * abs(e1[0])
            assert abs(res[k] - r1[0]) <= 1e3 * rtol * max(r1[0], 1e-3)


# tolerance in MeV, updates by which rounding at the threshold may move the stop
@pytest.mark.parametrize("prec,tol,slack", [(P.PNM_PREC_FP64, 1e-7, 0), (P.PNM_PREC_BF16X3, 1e-3, 1)])
def test_systems_converge_on_their_own(prec, tol, slack):
    # a system with few amplitudes, systems that converge at different updates
    N, rho, n2 = [14, 2, 14, 38], [0.08, 0.02, 0.2, 0.08], [9, 1, 12, 14]
    opts = dict(alpha=0.5, tol=tol, max_iter=200, precision=prec)
    with P.Context(N, rho, n2) as ctx:
        dE, it, _, _ = ctx.solve(**opts)
        for k in range(4):
            with P.Context(N[k], rho[k], n2[k]) as alone:
                e1, i1, _, _ = alone.solve(**opts)
            assert abs(int(it[k]) - int(i1[0])) <= slack
            assert abs(dE[k] - e1[0]) <= 2 * tol  # both within the stopping rule of the same fixed point
