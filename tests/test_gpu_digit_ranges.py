"""The ph term of FP64 accuracy on amplitudes of very different size: every cross channel has its own
scale, so that what lies in one channel costs the others no accuracy, and a channel whose rows or
columns lie too far apart for one scale is summed in FP64."""
import numpy as np
import pytest

import spinflip
from conftest import minnesota_params
from inputs import random_amplitudes
from oracle import channel

pytestmark = pytest.mark.gpu

# (neutrons, protons, density, n2max) with channels of more than eight rows, S_z = 0 and S_z > 0
SYSTEMS = [(38, 0, 0.12, 10), (66, 0, 0.16, 14), (14, 14, 0.16, 6)]
# two chained sums of at most 33 products and the four terms of an amplitude: 70 roundings of 2^-53, and of
# 2^-47 where pairs of 48 bits are summed
TOL, TOL_PAIR = 1e-14, 5e-13


@pytest.fixture(scope="module")
def pkg():
    from paper_1611_06765_gb300 import build
    build.build()
    import paper_1611_06765_gb300 as P
    return P


class Case:
    """A system, random flip-symmetric amplitudes with one of them scaled by `factor`, and which cross
    channels that one is in."""

    def __init__(self, pkg, N, Z, rho, n2, factor):
        P = minnesota_params()
        self.g = pkg.Context(N, rho, n2, params=P, Z=Z) if Z else pkg.Context(N, rho, n2, params=P)
        self.o = channel.OracleSystem(N, rho, n2, P, Z=Z)
        lab, st = self.g.amplitude_labels(), self.o.states()
        perm = spinflip.flip_permutation(lab, st)
        self.even = spinflip.symmetrise(random_amplitudes(len(lab), seed=9), perm)
        # one amplitude between states of the two channels every pair of states has: in the middle
        big = len(lab) // 3
        both = np.unique([big, perm[0][big]])
        self.t = self.even.copy()
        self.t[both] *= factor
        # keys of the four cross channels that each amplitude is an element of and reads from
        a, b, i, j = lab.T
        diff = np.stack([st[p] - st[h] for p, h in ((a, i), (a, j), (b, i), (b, j))], axis=1)
        self.sz0 = diff[:, :, 3] == 0
        self.key = np.ravel_multi_index(tuple((diff + 32).reshape(-1, diff.shape[2]).T), (65,) * diff.shape[2])
        _, self.key = np.unique(self.key, return_inverse=True)
        self.key = self.key.reshape(len(lab), 4)
        self.far = ~np.isin(self.key, np.unique(self.key[both]))  # channels without the scaled amplitude

    def tolerance(self, bound):
        """Per amplitude, in units of the relative error: its own sum of absolute products, of channels
        without the scaled amplitude the largest such sum in them (the scale of their digits), and of
        S_z = 0 channels with it the largest of all (they are formed from sums and differences of two
        blocks)."""
        apart = self.far.all(axis=1)
        top = np.zeros(self.key.max() + 1)
        np.maximum.at(top, self.key[apart].ravel(), np.repeat(bound[apart], 4))
        return bound + np.where(self.far, top[self.key], np.where(self.sz0, bound.max(), 0.0)).sum(axis=1)


@pytest.mark.parametrize("N,Z,rho,n2", SYSTEMS)
@pytest.mark.parametrize("factor", [2.0 ** 10, 2.0 ** 20, 2.0 ** 53])
def test_one_dominant_amplitude(pkg, N, Z, rho, n2, factor):
    c = Case(pkg, N, Z, rho, n2, factor)
    ref, bound = c.o.ph_apply(c.t), c.o.ph_apply(c.t, absval=True)
    tol = c.tolerance(bound)
    assert np.count_nonzero(c.far.all(axis=1)) > len(ref) // 2
    assert np.all(np.abs(c.g.apply_ph_term(c.t) - ref) <= TOL * tol)
    assert np.all(np.abs(c.g.apply_ph_term(c.t, precision=pkg.PNM_PREC_F32PAIR) - ref) <= TOL_PAIR * tol)
    c.g.close()


@pytest.mark.parametrize("N,Z,rho,n2", SYSTEMS)
def test_infinite_amplitude_stays_in_its_channels(pkg, N, Z, rho, n2):
    """The channels without it give the same bits whatever its value."""
    c = Case(pkg, N, Z, rho, n2, np.inf)
    apart = c.far.all(axis=1)
    for prec in (pkg.PNM_PREC_FP64, pkg.PNM_PREC_F32PAIR):
        r, plain = c.g.apply_ph_term(c.t, precision=prec), c.g.apply_ph_term(c.even, precision=prec)
        assert np.array_equal(r[apart], plain[apart])
        assert not np.all(np.isfinite(r[~apart])) and np.all(np.isfinite(plain))
    c.g.close()


@pytest.mark.parametrize("N,Z,rho,n2", SYSTEMS)
@pytest.mark.parametrize("alone", [False, True])
def test_large_amplitudes(pkg, N, Z, rho, n2, alone):
    """Amplitudes of a million, where the quadratic part is far above <kb|v|cj>, and one of 1e10 with zeros
    for the others, which meets <kb|v|cj> by itself."""
    c = Case(pkg, N, Z, rho, n2, 1.0)
    one, k = np.zeros_like(c.even), len(c.even) // 3
    idx, sign = spinflip.flip_permutation(c.g.amplitude_labels(), c.o.states())
    one[k] = 1e10
    one[idx[k]] = sign[k] * 1e10
    t = one if alone else 1e6 * c.even
    ref, bound = c.o.ph_apply(t), c.o.ph_apply(t, absval=True)
    tol = bound + (np.where(~c.far & c.sz0, bound.max(), 0.0).sum(axis=1) if alone else 0.0)
    assert np.all(np.abs(c.g.apply_ph_term(t) - ref) <= TOL * tol)
    assert np.all(np.abs(c.g.apply_ph_term(t, precision=pkg.PNM_PREC_F32PAIR) - ref) <= TOL_PAIR * tol)
    c.g.close()


@pytest.mark.parametrize("N,Z,rho,n2", SYSTEMS)
def test_pair_results_are_rounded(pkg, N, Z, rho, n2):
    """The ladder's sums are the same integers for both result types: a pair of FP32 numbers, rounded to 24
    bits and the rest to 24 more, is within 2^-49 of them, an FP64 number within 2^-53."""
    P = minnesota_params()
    g = pkg.Context(N, rho, n2, params=P, Z=Z) if Z else pkg.Context(N, rho, n2, params=P)
    t = random_amplitudes(len(g.amplitude_labels()), seed=13)
    r, pair = g.apply_pp_ladder(t), g.apply_pp_ladder(t, precision=pkg.PNM_PREC_F32PAIR)
    assert np.any(r) and np.all(np.abs(pair - r) <= 2.0 ** -48 * np.abs(r))
    g.close()


def _ladder(o, t):
    """(reference, sum of absolute products) of the pp ladder in the library's order."""
    tab = o.channel_tables()
    ref, bound, off = np.zeros(len(t)), np.zeros(len(t)), 0
    for c, (nh, npp) in enumerate(zip(tab["nhh"], tab["npp"])):
        s = slice(off, off + int(nh) * int(npp))
        off = s.stop
        V, tb = o.vpp_block(c), t[s].reshape(int(nh), int(npp))
        ref[s], bound[s] = (tb @ V).ravel(), (np.abs(tb) @ np.abs(V)).ravel()
    return ref, bound


@pytest.mark.parametrize("N,Z,rho,n2", [(2, 0, 0.3, 36), (14, 0, 0.3, 24), (38, 0, 0.12, 10), (2, 2, 0.2, 9),
                                           (14, 14, 0.2, 8)])
@pytest.mark.parametrize("kind", ["mbpt2", "random", "dominant", "single"])
def test_ladder_of_an_interaction_of_wide_range(pkg, N, Z, rho, n2, kind):
    """Every result against its own sum of absolute products.  The Gaussians exp(-x) of both sides carry an
    argument of three roundings, 4 x units of the last place with the function, x up to q^2 / 4 kappa_S at the
    largest momentum transfer 2 sqrt(n2max); sums of at most 900 products carry 900 more.  FP32 pairs, where the
    result is far from their smallest number, 2^-48."""
    P = minnesota_params()
    g = pkg.Context(N, rho, n2, params=P, Z=Z) if Z else pkg.Context(N, rho, n2, params=P)
    o = channel.OracleSystem(N, rho, n2, P, Z=Z)
    x = (2 * np.pi / o.L) ** 2 * 4 * n2 / (4 * P[5])
    tol = (4 * x + 900) * 2.0 ** -53
    t = random_amplitudes(len(g.amplitude_labels()), seed=31)
    k = np.flatnonzero(_ladder(o, t)[1])
    k = k[len(k) // 3]
    if kind == "mbpt2":
        g.mbpt3()
        t = g.get_amplitudes()
    elif kind == "dominant":
        t[k] = 2.0 ** 53
    elif kind == "single":
        t = np.zeros_like(t)
        t[k] = 1.0
    ref, bound = _ladder(o, t)
    assert np.all(np.abs(g.apply_pp_ladder(t) - ref) <= tol * bound)
    pair = g.apply_pp_ladder(t, precision=pkg.PNM_PREC_F32PAIR)
    seen = np.abs(ref) > 1e-20
    assert np.all(np.abs(pair - ref)[seen] <= ((tol + 2.0 ** -48) * bound)[seen])
    g.close()


@pytest.mark.parametrize("N,Z,rho,n2", [(2, 0, 0.3, 36), (14, 0, 0.3, 24), (38, 0, 0.3, 20), (2, 2, 0.2, 9)])
@pytest.mark.parametrize("single", [False, True])
def test_mixed_ladder_of_an_interaction_of_wide_range(pkg, N, Z, rho, n2, single):
    """V and t as BF16 hi + lo of their FP32 values, three products: 3 * 2^-18 of every product and the FP32
    sums of at most 500 terms, 2^-24 each; where the sum of absolute products is an ordinary FP32 number."""
    P = minnesota_params()
    g = pkg.Context(N, rho, n2, params=P, Z=Z) if Z else pkg.Context(N, rho, n2, params=P)
    o = channel.OracleSystem(N, rho, n2, P, Z=Z)
    g.mbpt3()
    t = g.get_amplitudes()
    if single:
        k = np.flatnonzero(_ladder(o, t)[1])
        t = np.zeros_like(t)
        t[k[len(k) // 3]] = 1.0
    ref, bound = _ladder(o, t)
    r = g.apply_pp_ladder(t, precision=pkg.PNM_PREC_BF16X3)
    seen = bound > 1e-30
    assert np.all(np.abs(r - ref)[seen] <= ((3 * 2.0 ** -18 + 500 * 2.0 ** -24) * bound)[seen])
    g.close()


def test_steep_and_ordinary_systems_in_one_context(pkg):
    """Only the systems whose interaction is steep have V in FP64 and their results checked in a solve: the
    same arithmetic per system as in contexts of their own, so the same bits but for the order of the energy
    sums, which end the iteration; 12 updates for all."""
    Ns, rhos, n2 = [2, 14, 14], [0.3, 0.08, 0.3], [24, 9, 24]
    kw = dict(alpha=0.5, tol=1e-300, max_iter=12, allow=(pkg.PNM_ENOTCONV,))
    g = pkg.Context(Ns, rhos, n2)
    g.solve(**kw)
    for k in range(3):
        one = pkg.Context(Ns[k], rhos[k], n2[k])
        one.solve(**kw)
        t, ref = g.get_amplitudes(k), one.get_amplitudes()
        assert np.all(np.abs(t - ref) <= 1e-13 * np.abs(ref))
        a = random_amplitudes(len(t), seed=k)
        assert np.array_equal(g.apply_pp_ladder(a, sys=k), one.apply_pp_ladder(a))
        one.close()
    g.close()
