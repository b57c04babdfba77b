"""The digit products of the pp ladder and the ph term (FP64 accuracy on the tensor cores) at the
sizes where they can go wrong: single steps and blocks, remainders along every dimension, one to
eight rows per pass and several passes, channels on both sides of the warp, tiny and CTA paths,
and amplitudes that are zero, tiny, huge, spread over many magnitudes, infinite or NaN."""
import numpy as np
import pytest

import spinflip
from conftest import minnesota_params
from inputs import random_amplitudes
from oracle import channel

pytestmark = pytest.mark.gpu

# (neutrons, protons, density, n2max): 1 x 1 blocks; ladder bases of 1-4 steps, up to 17 rows per
# channel; ph channels of 1-33 rows and columns
SYSTEMS = [(2, 0, 0.08, 1), (2, 0, 0.08, 9), (14, 0, 0.08, 2), (14, 0, 0.08, 9), (38, 0, 0.12, 4), (54, 0, 0.12, 8),
           (66, 0, 0.16, 6), (66, 0, 0.16, 14), (2, 2, 0.16, 3), (14, 14, 0.16, 6)]


@pytest.fixture(scope="module")
def pkg():
    from paper_1611_06765_gb300 import build
    build.build()
    import paper_1611_06765_gb300 as P
    return P


def _pair(pkg, N, Z, rho, n2):
    P = minnesota_params()
    if Z:
        return pkg.Context(N, rho, n2, params=P, Z=Z), channel.OracleSystem(N, rho, n2, P, Z=Z)
    return pkg.Context(N, rho, n2, params=P), channel.OracleSystem(N, rho, n2, P)


def _ladder(o, t):
    """(reference, sum of absolute products) of the pp ladder in the library's order."""
    tab = o.channel_tables()
    ref, bound, off = np.zeros(len(t)), np.zeros(len(t)), 0
    for c, (nh, npp) in enumerate(zip(tab["nhh"], tab["npp"])):
        s = slice(off, off + int(nh) * int(npp))
        off = s.stop
        V, tb = o.vpp_block(c), t[s].reshape(int(nh), int(npp))
        with np.errstate(invalid="ignore", over="ignore"):
            ref[s], bound[s] = (tb @ V).ravel(), (np.abs(tb) @ np.abs(V)).ravel()
    return ref, bound


@pytest.mark.parametrize("N,Z,rho,n2", SYSTEMS)
@pytest.mark.parametrize("spread", [0, 12])
def test_operators_against_oracle(pkg, N, Z, rho, n2, spread):
    """Both sides sum at most 900 FP64 products whose interaction elements agree to a few units of
    the last place; the digit kernel's own terms are below 2^-60 of the product of the largest
    values.  1e-14 of the largest sum of absolute products covers the sums of both."""
    g, o = _pair(pkg, N, Z, rho, n2)
    n = len(g.amplitude_labels())
    t = random_amplitudes(n, seed=21)
    if spread:
        t = t * 10.0 ** -np.random.default_rng(5).uniform(0, spread, n)
    ref, bound = _ladder(o, t)
    tol = 1e-14 * max(np.max(bound), 1e-300)
    assert np.max(np.abs(g.apply_pp_ladder(t) - ref)) <= tol
    assert np.max(np.abs(g.apply_pp_ladder(t, precision=pkg.PNM_PREC_F32PAIR) - ref)) <= tol
    perm = spinflip.flip_permutation(g.amplitude_labels(), o.states()) if not Z else None
    if perm is not None:
        ts = spinflip.symmetrise(t, perm)
        ref, bound = o.ph_apply(ts), o.ph_apply(ts, absval=True)
        tol = 1e-14 * max(np.max(bound), 1e-300)
        assert np.max(np.abs(g.apply_ph_term(t) - ref)) <= tol
        # FP32 pairs of the smallest channels carry 48 bits
        assert np.max(np.abs(g.apply_ph_term(t, precision=pkg.PNM_PREC_F32PAIR) - ref)) <= 10 * tol
    g.close()


@pytest.mark.parametrize("N,Z,rho,n2", [s for s in SYSTEMS if not s[1]])
def test_mixed_ph_operator(pkg, N, Z, rho, n2):
    """The FP32 ph term over channels of 1 to 33 rows and columns (a part of a warp, a warp, a CTA each):
    two chained FP32 products over at most 33 terms, 2 * 33 * 2^-24 < 4e-6 of the element's sum of
    absolute products, and the rounding of the operands, 3 * 2^-24."""
    g, o = _pair(pkg, N, Z, rho, n2)
    t = random_amplitudes(len(g.amplitude_labels()), seed=17)
    ts = spinflip.symmetrise(t, spinflip.flip_permutation(g.amplitude_labels(), o.states()))
    ref, bound = o.ph_apply(ts), o.ph_apply(ts, absval=True)
    assert np.all(np.abs(g.apply_ph_term(t, precision=pkg.PNM_PREC_BF16X3) - ref) <= 5e-6 * bound + 1e-30)
    g.close()


@pytest.mark.parametrize("N,Z,rho,n2", [(14, 0, 0.08, 9), (66, 0, 0.16, 14), (14, 14, 0.16, 6)])
def test_power_of_two_scaling_is_exact(pkg, N, Z, rho, n2):
    """The ladder is linear and its digits carry one exponent per row: scaled amplitudes give the
    scaled result bit for bit, down to values whose products leave the normal range."""
    g, _ = _pair(pkg, N, Z, rho, n2)
    t = random_amplitudes(len(g.amplitude_labels()), seed=3)
    r = g.apply_pp_ladder(t)
    for k in (-900, -40, 13, 900):
        assert np.array_equal(g.apply_pp_ladder(np.ldexp(t, k)), np.ldexp(r, k))
    assert not np.any(g.apply_pp_ladder(np.zeros_like(t)))
    assert not np.any(g.apply_ph_term(np.zeros_like(t)))
    tiny = g.apply_ph_term(np.ldexp(t, -900))  # linear part only: the quadratic one is below it
    lin = g.apply_ph_term(np.ldexp(t, -200))
    assert np.max(np.abs(np.ldexp(tiny, 700) - lin)) <= 2.0 ** -50 * np.max(np.abs(lin))
    g.close()


@pytest.mark.parametrize("N,n2", [(14, 9), (66, 14)])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_amplitudes(pkg, N, n2, bad):
    """One non-finite amplitude: its row of the ladder is what FP64 arithmetic gives (infinities
    with their sign, NaN), every other row is unchanged bit for bit; the ph term is non-finite
    somewhere and a solve started from it ends as diverged."""
    g, o = _pair(pkg, N, 0, 0.16, n2)
    t = random_amplitudes(len(g.amplitude_labels()), seed=4)
    r = g.apply_pp_ladder(t)
    tab = o.channel_tables()
    off, c = 0, int(np.argmax(tab["npp"] * (np.abs(r).sum() > 0)))
    sizes = tab["nhh"].astype(int) * tab["npp"].astype(int)
    for c in np.argsort(-sizes):
        off = int(sizes[:c].sum())
        if np.any(r[off:off + sizes[c]]):
            break
    npp = int(tab["npp"][c])
    t[off + 2] = bad
    ref, _ = _ladder(o, t)
    rb = g.apply_pp_ladder(t)
    row = slice(off, off + npp)
    assert np.array_equal(np.isnan(rb[row]), np.isnan(ref[row]))
    assert np.array_equal(rb[row][np.isinf(ref[row])], ref[row][np.isinf(ref[row])])
    keep = np.ones(len(t), bool)
    keep[row] = False
    assert np.array_equal(rb[keep], r[keep])
    assert not np.all(np.isfinite(g.apply_ph_term(t)))
    g.set_amplitudes(t)
    _, _, _, rc = g.solve(alpha=0.5, tol=1e-8, max_iter=20, init=pkg.PNM_INIT_KEEP, allow=(pkg.PNM_EDIVERGED,))
    assert rc == pkg.PNM_EDIVERGED
    g.close()
