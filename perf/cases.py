"""The work that users of this library have it do, for timing and for comparing results.

A case is one call (or one short fixed sequence of calls) of the public interface in
``paper_1611_06765_gb300`` on a physical system (N neutrons and Z protons per box, density,
plane waves with n^2 <= n2max, optionally a batch of densities or a twist mesh):

  solve    a CCD solve from the MBPT2 start to the stopping rule, energies, update counts and the
           converged amplitudes read back (FP64, or mixed precision with refinement sweeps)
  mbpt3    the three third-order diagrams
  create   a context built from scalars, its reference and second-order energies
  pp, ph   the pp-ladder and ph terms as operators on host amplitudes
  predict  the learned start written into the held amplitudes and read back
  grad     loss and gradient of the warm-start network on one training batch

The densities are the configurations' own, moved by up to 2% by the seed.  Results of the mixed
mode (BF16x3 / FP32 contractions) and of the BF16 network are handed on in FP32, the type those
contractions accumulate in: their last bits depend on the split of the sums that the library's
tile tuner picks by timing, and a consumer (the network's training set) takes them in FP32.
``exact`` is a restatement in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

MIX = dict(alpha=0.5, tol=1e-30, max_iter=500)
SHELLS = {2: 1, 14: 2, 38: 3, 54: 4, 66: 5}  # closed shells of neutrons: the smallest n2max that leaves particles
HELDOUT3 = (0.05, 0.11, 0.17)
F, H = 32, 128  # warm-start network: features, hidden width


def listed():
    return [
        # the smallest system of the test suite and the smoke test: 66 states, all latency
        dict(name="solve_n14_n4_fp64", do="solve", N=14, rho=0.08, n2max=4, batch=1, prec="fp64", tol_N=1e-11),
        # one N = 14 density in mixed precision: launches and short kernels
        dict(name="solve_n14_n20_mixed", do="solve", N=14, rho=0.08, n2max=20, batch=1, prec="mixed", tol_N=1e-6),
        # the default precision on the paper's table of N = 66, n^2 <= 42 (2378 states)
        dict(name="solve_n66_n42_fp64", do="solve", N=66, rho=0.08, n2max=42, batch=1, prec="fp64", tol_N=1e-6),
        # the benchmark's batch of three densities, mixed precision, two FP32-pair sweeps
        dict(name="solve_n66_n36_x3_mixed", do="solve", N=66, rho=0.11, n2max=36, batch=3, prec="mixed", tol_N=1e-6),
        # symmetric nuclear matter, 14 + 14, FP64: over a hundred updates of mid-size channels
        dict(name="solve_snm28_n20_fp64", do="solve", N=14, Z=14, rho=0.16, n2max=20, batch=1, prec="fp64", tol_N=1e-6),
        # twist averaging: 120 small systems in one context
        dict(name="solve_n14_twist120_mixed", do="solve", N=14, rho=0.08, n2max=20, mesh="4x5x6", prec="mixed", tol_N=1e-6),
        # third order for three densities at once
        dict(name="mbpt3_n66_n36_x3", do="mbpt3", N=66, rho=0.11, n2max=36, batch=3),
        # a new context and its second-order energies: what a scan over densities pays per point
        dict(name="create_n66_n36_x3", do="create", N=66, rho=0.11, n2max=36, batch=3),
        # the ladder as an operator inside a user's own iteration, FP32-pair kernels
        dict(name="pp_n66_n36_pair", do="pp", N=66, rho=0.16, n2max=36, batch=1, prec="pair"),
        # the particle-hole term as an operator, mixed-precision kernels
        dict(name="ph_n66_n36_mixed", do="ph", N=66, rho=0.16, n2max=36, batch=1, prec="mixed"),
        # the learned start of the benchmark's batch
        dict(name="predict_n66_n36_x3", do="predict", N=66, rho=0.11, n2max=36, batch=3),
        # one training batch of the warm-start network, forward and backward, BF16
        dict(name="grad_1024", do="grad", rows=1024, prec="bf16"),
    ]


def draw(rng):
    do = rng.choice(("solve", "solve", "solve", "mbpt3", "create", "pp", "ph", "predict", "grad"))
    if do == "grad":
        return dict(do=do, rows=int(round(math.exp(rng.uniform(math.log(33), math.log(8192))))),
                    prec=rng.choice(("bf16", "bf16", "simt", "fp32")))
    N = rng.choice((2, 14, 14, 38, 54, 66))
    lo, hi = SHELLS[N], 36 if N > 14 else 24
    c = dict(do=do, N=N, rho=round(math.exp(rng.uniform(math.log(0.02), math.log(0.3))), 4),
             n2max=int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))
    c["batch"] = rng.randint(1, 3) if N > 14 else int(round(math.exp(rng.uniform(0, math.log(16)))))
    if do == "solve":
        c["prec"] = rng.choice(("fp64", "mixed", "mixed64"))
        c["tol_N"] = 1e-6
        if c["prec"] == "fp64":
            c["tol_N"] = rng.choice((1e-6, 1e-8))
            c["batch"] = c["batch"] if N <= 14 else 1
            if rng.random() < 0.4:
                c["terms"] = rng.choice((1, 2, 3))
        if N == 14 and rng.random() < 0.3:
            c["mesh"], c["batch"] = rng.choice(("1x2x4", "2x3x4")), 1
        elif N in (2, 14) and rng.random() < 0.3:
            c.update(Z=N, batch=1, n2max=min(c["n2max"], 18), rho=round(rng.uniform(0.12, 0.2), 4), tol_N=1e-6)
            c.pop("terms", None)
    elif do in ("pp", "ph"):
        c["prec"], c["batch"] = rng.choice(("fp64", "pair", "mixed")), 1
    return c


# ------------------------------------------------------------------ what a user's program does
def _rng(seed, k=0):
    return np.random.default_rng([seed & 0x7FFFFFFF, k])


def _systems(case, seed):
    """(N, Z or None, densities, n2max, twists or None) of the case's context."""
    move = 1.0 + 0.02 * _rng(seed).uniform(-1.0, 1.0)
    if case.get("mesh"):
        theta = _mesh(case["mesh"])
        return case["N"], case.get("Z"), [case["rho"] * move] * len(theta), case["n2max"], theta
    n = case.get("batch", 1)
    if n == 3 and case["rho"] == 0.11:
        rhos = [r * move for r in HELDOUT3]
    else:
        rhos = [case["rho"] * move * (1.0 + 0.05 * k) for k in range(n)]
    return case["N"], case.get("Z"), rhos, case["n2max"], None


def _mesh(text):
    """Gauss-Legendre nodes on [0, pi], x-major."""
    ax = [0.5 * math.pi * (np.polynomial.legendre.leggauss(int(k))[0] + 1.0) for k in text.split("x")]
    return np.stack([g.ravel() for g in np.meshgrid(*ax, indexing="ij")], axis=1)


def _network(seed):
    """Parameters in the library's order, and their parts by name: weights of a trained
    network's size, He-scaled; the output a small correction of the MBPT2 amplitudes."""
    r = _rng(seed, 1)
    p = dict(mu=r.normal(0, 0.1, F), istd=r.uniform(0.8, 1.2, F), ys=np.array([0.1]), pad=np.zeros(3),
             w1=r.normal(0, math.sqrt(2 / F), (H, F)), b1=r.normal(0, 0.1, H), w2=r.normal(0, math.sqrt(2 / H), (H, H)),
             b2=r.normal(0, 0.1, H), w3=r.normal(0, math.sqrt(2 / H), (H, H)), b3=r.normal(0, 0.1, H),
             w4=r.normal(0, math.sqrt(1 / H), H), b4=r.normal(0, 0.1, 1))
    p = {k: v.astype(np.float32) for k, v in p.items()}
    return np.concatenate([v.ravel() for v in p.values()]), p


def _batch(case, seed):
    r = _rng(seed, 2)
    X = r.normal(0, 1, (case["rows"], F)).astype(np.float32)
    X[:, 22:] = 0
    return X, r.normal(0, 1, case["rows"]).astype(np.float32)


def _amplitudes(n, seed):
    return _rng(seed, 3).normal(0.0, 0.05, n)


def prepare(case, seed):
    import paper_1611_06765_gb300 as P
    state = dict(P=P, case=case)
    if case["do"] == "grad":
        state["blob"], _ = _network(seed)
        state["X"], state["T"] = _batch(case, seed)
        return state
    N, Z, rhos, n2, theta = _systems(case, seed)
    state["args"] = dict(N=N, rho=rhos, n2max=n2, theta=theta, Z=Z)
    if case["do"] == "create":
        return state
    state["ctx"] = P.Context(**state["args"])
    if case["do"] in ("pp", "ph"):
        state["t"] = _amplitudes(len(state["ctx"].get_amplitudes(0)), seed)
    if case["do"] == "predict":
        state["ctx"].mlp_set_model(_network(seed)[0])
    return state


def _fp32(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(torch.float32)


def run(state):
    P, case = state["P"], state["case"]
    do, prec = case["do"], case.get("prec")
    if do == "grad":
        loss, g = P.mlp_loss_grad(state["blob"], state["X"], state["T"], fp32=prec == "fp32", tensor_cores=prec == "bf16")
        return dict(loss=np.float32(loss), grad=g)
    if do == "create":
        ctx = P.Context(**state["args"])
        eref, e2 = ctx.eref(), ctx.mbpt2()
        _, eps, _ = ctx.basis(0)
        ctx.close()
        return dict(eref=eref, mbpt2=e2, eps=eps)
    ctx = state["ctx"]
    if do == "mbpt3":
        return dict(e3=ctx.mbpt3())
    if do == "predict":
        ctx.mlp_predict()
        return dict(t=torch.cat([_fp32(ctx.get_amplitudes(k)) for k in range(ctx.nsys)]))
    if do in ("pp", "ph"):
        how = dict(fp64=P.PNM_PREC_FP64, pair=P.PNM_PREC_F32PAIR, mixed=P.PNM_PREC_BF16X3)[prec]
        r = (ctx.apply_pp_ladder if do == "pp" else ctx.apply_ph_term)(state["t"], precision=how)
        return dict(r=_fp32(r) if prec == "mixed" else r)
    kw = dict(MIX, tol_per_N=case["tol_N"])
    if prec != "fp64":
        kw.update(precision=P.PNM_PREC_BF16X3, refine_sweeps=2,
                  refine_kernels=P.PNM_PREC_F32PAIR if prec == "mixed" else P.PNM_PREC_FP64)
    # a density without a fixed point in reach is an ordinary answer of a scan
    dE, it, _, rc = ctx.solve(terms=case.get("terms", 0), allow=(P.PNM_ENOTCONV, P.PNM_EDIVERGED), **kw)
    as_read = torch.from_numpy if prec == "fp64" else _fp32
    return dict(dE=as_read(dE), t=torch.cat([as_read(ctx.get_amplitudes(k)) for k in range(ctx.nsys)]), iters=it, rc=rc)


# ------------------------------------------------------------------------- in 64 bits, in torch
VR, KR, VT, KT, VS, KS, H2M = 200.0, 1.487, -178.0, 0.639, -91.85, 0.465, 20.721  # Minnesota, MeV and fm


class System:
    """One box in plain torch: states, restricted pairs per conserved momentum and charge in the
    library's order, and the terms of the CCD equations."""

    def __init__(self, N, Z, rho, n2max, theta=None):
        dev = self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.A, self.rho = N + (Z or 0), rho
        species = [t for t, k in ((-1, Z or 0), (1, N)) if k]
        r = int(math.isqrt(n2max))
        ax = np.arange(-r, r + 1)
        n = np.stack([g.ravel() for g in np.meshgrid(ax, ax, ax, indexing="ij")], axis=1)
        n2 = (n * n).sum(1)
        n = n[n2 <= n2max][np.argsort(n2[n2 <= n2max], kind="stable")]
        sp = [(s, t) for s in (-1, 1) for t in species]
        st = np.concatenate([np.repeat(n, len(sp), axis=0), np.tile(np.array(sp), (len(n), 1))], axis=1)
        phi = np.zeros(3) if theta is None else np.asarray(theta) / (2 * math.pi)
        k2 = np.sort((st[:, :3] + phi) ** 2, axis=1)
        k2 = (k2[:, 0] + k2[:, 1]) + k2[:, 2]
        if theta is not None:
            o = np.argsort(k2, kind="stable")
            st, k2 = st[o], k2[o]
        self.L = (self.A / rho) ** (1 / 3)
        self.st = st
        self.s = torch.as_tensor(st, device=dev)
        m = torch.arange(4 * n2max + 1, device=dev, dtype=torch.float64) * (2 * math.pi / self.L) ** 2
        self.lut = torch.stack([0.5 * v / self.L ** 3 * (math.pi / k) ** 1.5 * torch.exp(-m / (4 * k))
                                for v, k in ((VR, KR), (VT, KT), (VS, KS))])
        nsp, A = len(st), self.A
        self.ekin = torch.as_tensor(H2M * (2 * math.pi / self.L) ** 2 * k2, device=dev)
        p, i = torch.arange(nsp, device=dev)[:, None], torch.arange(A, device=dev)[None, :]
        self.eps = self.ekin + self.v(p, i, p, i).sum(1)
        self.eref = float(0.5 * (self.ekin[:A].sum() + self.eps[:A].sum()))
        self.mm, self.nq = 2 * r, 3 if Z in (None, 0) else 9
        self._direct(nsp, A)

    def v(self, p, q, r, s):
        """Antisymmetrized <pq|v|rs> of momentum-conserving, broadcastable index arrays."""
        P, Q, R, S = (self.s[x] for x in (p, q, r, s))
        e = lambda x, y, c: x[..., c] == y[..., c]  # noqa: E731
        sd, sx = e(P, R, 3) & e(Q, S, 3), e(P, S, 3) & e(Q, R, 3)
        td, tx = e(P, R, 4) & e(Q, S, 4), e(P, S, 4) & e(Q, R, 4)
        one, ps, pt, pst = ((a & b).double() for a, b in ((sd, td), (sx, td), (sd, tx), (sx, tx)))
        m1, m2 = ((x[..., :3] - y[..., :3]).square().sum(-1) for x, y in ((P, R), (P, S)))
        out = 0.0
        for c, lut in zip((2 * (one - pst), one + ps - pt - pst, one - ps + pt - pst), self.lut):
            out = out + c * (lut[m1] + lut[m2])
        return 0.5 * out

    def _key(self, q):
        m, M = self.mm, 2 * self.mm + 1
        slot = (q[:, 3] + 2) // 2
        if self.nq == 9:
            slot = 3 * slot + (q[:, 4] + 2) // 2
        return (((q[:, 0] + m) * M + q[:, 1] + m) * M + q[:, 2] + m) * self.nq + slot

    def _direct(self, nsp, A):
        dev, st = self.dev, self.st

        def pairs(lo, hi):
            a, b = np.triu_indices(hi - lo, 1)
            a, b = a + lo, b + lo
            k = self._key(st[a] + st[b])
            o = np.argsort(k, kind="stable")
            return a[o], b[o], k[o]

        hi, hj, hk = pairs(0, A)
        pa, pb, pk = pairs(A, nsp)
        keys = np.intersect1d(hk, pk)
        h0, h1 = np.searchsorted(hk, keys), np.searchsorted(hk, keys, "right")
        p0, p1 = np.searchsorted(pk, keys), np.searchsorted(pk, keys, "right")
        self.nh, self.np_ = h1 - h0, p1 - p0
        self.off = np.concatenate([[0], np.cumsum(self.nh * self.np_)])
        self.n = int(self.off[-1])
        slot = keys % self.nq  # identical nucleons of equal spin do not interact
        self.lad = slot == 1 if self.nq == 3 else (slot // 3 == 1) | (slot % 3 == 1)
        posh, posp = np.full((nsp, nsp), -1), np.full((nsp, nsp), -1)
        chan = np.full((A, A), -1)
        T = lambda x: torch.as_tensor(x, device=dev)  # noqa: E731
        self.ch = []
        lab = [[], [], [], []]
        for c in range(len(keys)):
            i, j, a, b = hi[h0[c]:h1[c]], hj[h0[c]:h1[c]], pa[p0[c]:p1[c]], pb[p0[c]:p1[c]]
            posh[i, j], posp[a, b], chan[i, j] = np.arange(len(i)), np.arange(len(a)), c
            self.ch.append((T(i), T(j), T(a), T(b)))
            for dst, x in zip(lab, (np.tile(a, len(i)), np.tile(b, len(i)), np.repeat(i, len(a)), np.repeat(j, len(a)))):
                dst.append(x)
        self.a, self.b, self.i, self.j = (T(np.concatenate(x)) if x else T(np.zeros(0, int)) for x in lab)
        self.posh, self.posp, self.chan = T(posh), T(posp), T(chan)
        self.toff, self.tnp = T(self.off), T(self.np_)
        self.vt = self.v(self.a, self.b, self.i, self.j)
        self.den = self.eps[self.i] + self.eps[self.j] - self.eps[self.a] - self.eps[self.b]
        self.t0 = self.vt / self.den

    def code(self, a, b, i, j):
        """(index, sign) of t_ij^ab for any order of the arguments; index n where it vanishes."""
        a, b, i, j = torch.broadcast_tensors(a, b, i, j)
        sign = torch.where(a > b, -1.0, 1.0) * torch.where(i > j, -1.0, 1.0)
        a, b = torch.minimum(a, b), torch.maximum(a, b)
        i, j = torch.minimum(i, j), torch.maximum(i, j)
        c = self.chan[i, j]
        z = self.toff[c] + self.posh[i, j] * self.tnp[c] + self.posp[a, b]
        return torch.where((a == b) | (i == j) | (c < 0), torch.full_like(z, self.n), z), sign

    def flip(self):
        """(index, sign) of every amplitude's partner under the flip of all spins."""
        where = {tuple(x): k for k, x in enumerate(self.st.tolist())}
        f = torch.as_tensor([where[(x, y, z, -s, q)] for x, y, z, s, q in self.st.tolist()], device=self.dev)
        return self.code(f[self.a], f[self.b], f[self.i], f[self.j])

    def blocks(self, t, c):
        return t[self.off[c]:self.off[c + 1]].view(int(self.nh[c]), int(self.np_[c]))

    def pp(self, t):
        out = torch.zeros_like(t)
        if not hasattr(self, "vpp"):
            self.vpp = {}
            for c in np.nonzero(self.lad)[0]:
                _, _, a, b = self.ch[c]
                self.vpp[c] = self.v(a[:, None], b[:, None], a[None], b[None])
        for c, V in self.vpp.items():
            self.blocks(out, c).copy_(self.blocks(t, c) @ V)
        return out

    def hh(self, t, chi=True):
        """hh ladder with <kl|chi|ij> (chi) or the bare interaction."""
        out = torch.zeros_like(t)
        if not hasattr(self, "vhh"):
            self.vhh = [self.v(i[:, None], j[:, None], i[None], j[None]) for i, j, _, _ in self.ch]
        for c, V in enumerate(self.vhh):
            x = self.blocks(t, c)
            if chi:
                V = V + self.blocks(self.vt, c) @ x.T
            self.blocks(out, c).copy_(V.T @ x)
        return out

    def one(self, t):
        """(d_a + d_b - d_i - d_j) t with the diagonal one-body intermediates."""
        vt, d = self.vt * t, torch.zeros(len(self.st), device=self.dev, dtype=torch.float64)
        for x, s in ((self.a, -1.0), (self.b, -1.0), (self.i, 1.0), (self.j, 1.0)):
            d.index_add_(0, x, s * vt)
        return (d[self.a] + d[self.b] - d[self.i] - d[self.j]) * t

    def _cross(self):
        A, nsp, st, dev = self.A, len(self.st), self.st, self.dev
        a, i = (g.ravel() for g in np.meshgrid(np.arange(A, nsp), np.arange(A), indexing="ij"))
        k, c = (g.ravel() for g in np.meshgrid(np.arange(A), np.arange(A, nsp), indexing="ij"))
        kr, kc = self._key(st[a] - st[i]), self._key(st[k] - st[c])
        keys = np.intersect1d(kr, kc)

        def rows(p, h, key):  # (channel, position) of every pair, and the padded lists per channel
            o = np.argsort(key, kind="stable")
            o = o[np.isin(key[o], keys)]
            x = np.searchsorted(keys, key[o])
            pos = np.arange(len(o)) - np.searchsorted(x, x)
            lst = np.full((2, len(keys), pos.max() + 1 if len(o) else 1), -1)
            lst[0, x, pos], lst[1, x, pos] = p[o], h[o]
            ch, at = np.full((nsp, A), -1), np.zeros((nsp, A), int)
            ch[p[o], h[o]], at[p[o], h[o]] = x, pos
            return [torch.as_tensor(u, device=dev) for u in (lst[0], lst[1], ch, at)]

        ra, ri, self.xch, self.xrow = rows(a, i, kr)
        cc, ck, _, self.xcol = rows(c, k, kc)
        R, C = ra.shape[1], cc.shape[1]
        row, col = (ra >= 0)[:, :, None], (cc >= 0)[:, None, :]
        # T[(a,i)][(k,c)] = t_ik^ac
        z, sg = self.code(ra.clamp(min=0)[:, :, None], cc.clamp(min=0)[:, None, :], ri.clamp(min=0)[:, :, None], ck.clamp(min=0)[:, None, :])
        self.xz = torch.where(row & col, z, torch.full_like(z, self.n))
        self.xs = sg
        q = [u.clamp(min=0) for u in (ra, ri, cc, ck)]
        both = (cc >= 0)[:, :, None] & col
        chunk = max(1, (1 << 24) // max(1, C * max(R, C)))
        self.v1 = torch.empty(len(keys), C, C, device=dev, dtype=torch.float64)
        self.w = torch.empty(len(keys), C, R, device=dev, dtype=torch.float64)
        for x in range(0, len(keys), chunk):
            e, l, c1, k1 = (u[x:x + chunk] for u in q)
            # <kb|v|cj> and <kl|v|ce>
            self.v1[x:x + chunk] = self.v(k1[:, :, None], c1[:, None, :], c1[:, :, None], k1[:, None, :]) * both[x:x + chunk]
            self.w[x:x + chunk] = self.v(k1[:, :, None], l[:, None, :], c1[:, :, None], e[:, None, :]) * (row & col)[x:x + chunk].transpose(1, 2)
        self.qz = []
        for a_, i_, j_, b_, s in ((self.a, self.i, self.j, self.b, 1.0), (self.a, self.j, self.i, self.b, -1.0),
                                  (self.b, self.i, self.j, self.a, -1.0), (self.b, self.j, self.i, self.a, 1.0)):
            x = self.xch[a_, i_]
            self.qz.append((torch.where(x >= 0, (x * R + self.xrow[a_, i_]) * C + self.xcol[b_, j_],
                                        torch.full_like(x, len(keys) * R * C)), s))

    def ph(self, t, linear=False):
        if not hasattr(self, "xz"):
            self._cross()
        zero = torch.zeros(1, device=self.dev, dtype=torch.float64)
        T = torch.cat([t, zero])[self.xz] * self.xs
        C = self.v1 if linear else self.v1 + 0.5 * torch.bmm(self.w, T)
        Q = torch.cat([torch.bmm(T, C).reshape(-1), zero])
        return sum(s * Q[z] for z, s in self.qz)

    def step(self, t, terms=0):
        x = self.vt + self.pp(t)
        if terms != 1:
            x = x + self.hh(t, chi=terms == 0)
        if terms in (0, 3):
            x = x + self.ph(t, linear=terms == 3)
        if terms == 0:
            x = x + self.one(t)
        return 0.5 * x / self.den + 0.5 * t

    def solve(self, tol, terms, sweeps, cap=500):
        t, e = self.t0, float((self.vt * self.t0).sum())
        left = -1
        for it in range(1, cap + sweeps + 1):
            t = self.step(t, terms)
            new = float((self.vt * t).sum())
            done, e = abs(new - e) < tol, new
            if left < 0 and (done or it == cap):
                left = sweeps
            elif left > 0:
                left -= 1
            if left == 0 and (done or not sweeps):
                break
        return e, t

    def features(self):
        kF = (3 * math.pi ** 2 * self.rho) ** (1 / 3)
        eF, s = H2M * kF * kF, self.s.double()
        X = torch.zeros(self.n, F, device=self.dev, dtype=torch.float64)
        for c, p in enumerate((self.a, self.b, self.i, self.j)):
            X[:, 3 * c:3 * c + 3] = 2 * math.pi / self.L / kF * s[p, :3]
            X[:, 12 + c] = s[p, 3]
        sigma = self.t0.square().mean().sqrt()
        X[:, 16], X[:, 17], X[:, 18] = self.den / eF, self.vt * self.A / eF, self.t0 / sigma
        X[:, 19], X[:, 20], X[:, 21] = self.rho / 0.16, kF, self.A / 66
        return X, sigma


def _net(p, X):
    h = (X - p["mu"]) * p["istd"]
    for k in "123":
        h = torch.nn.functional.gelu(h @ p["w" + k].T + p["b" + k], approximate="tanh")
    return h @ p["w4"] + p["b4"]


def exact(case, seed):
    do = case["do"]
    if do == "grad":
        X, T = _batch(case, seed)
        p = {k: torch.from_numpy(v).double().requires_grad_(k[0] in "wb") for k, v in _network(seed)[1].items()}
        loss = (_net(p, torch.from_numpy(X).double()) - torch.from_numpy(T).double()).square().mean()
        loss.backward()
        g = torch.cat([(v.grad if v.grad is not None else torch.zeros_like(v)).reshape(-1) for v in p.values()])
        return dict(loss=loss.detach(), grad=g)
    N, Z, rhos, n2, theta = _systems(case, seed)
    if theta is not None:
        return None  # one system after the other: over 20 seconds
    if len(rhos) > 4:
        return None
    sys = [System(N, Z, r, n2) for r in rhos]
    if do == "create":
        return dict(eref=np.array([s.eref for s in sys]), mbpt2=np.array([float((s.vt * s.t0).sum()) for s in sys]),
                    eps=sys[0].eps)
    if do == "mbpt3":
        return dict(e3=torch.stack([torch.stack([(s.t0 * x).sum() for x in (s.pp(s.t0), s.hh(s.t0, False), s.ph(s.t0, True))])
                                    for s in sys]))
    if do in ("pp", "ph"):
        s = sys[0]
        t = torch.as_tensor(_amplitudes(s.n, seed), device=s.dev)
        if do == "pp":
            return dict(r=s.pp(t))
        z, sign = s.flip()  # the term of the flip-symmetric part
        return dict(r=s.ph(0.5 * (t + sign * t[z])))
    if do == "predict":
        p = {k: torch.as_tensor(v, device=sys[0].dev).double() for k, v in _network(seed)[1].items()}
        out = []
        for s in sys:
            X, sigma = s.features()
            y = s.t0 + sigma * p["ys"] * _net(p, X)
            # evaluated on the first amplitude of each spin-flip pair and copied to the other
            z, sign = s.flip()
            out.append(torch.where(z < torch.arange(s.n, device=s.dev), sign * y[z], y))
        return dict(t=torch.cat(out))
    got = []
    for s in sys:
        got.append(s.solve(case["tol_N"] * s.A, case.get("terms", 0), 0 if case["prec"] == "fp64" else 2))
        for x in ("vpp", "vhh", "v1", "w", "xz", "xs", "qz"):
            s.__dict__.pop(x, None)
    return dict(dE=np.array([e for e, _ in got]), t=torch.cat([t for _, t in got]), iters=None, rc=None)


# ------------------------------------------------------------------------------------ work
def _counts(N, Z, n2max):
    """Per system: amplitudes, flops of one pp ladder, of one hh ladder and of one ph term (spin
    symmetries used), elements of the pp interaction and of the cross channels."""
    s = System(N, Z, 0.16, n2max)
    nh, npp, A, st = s.nh.astype(float), s.np_.astype(float), s.A, s.st
    # two neutrons of opposite spin interact in the singlet only: half as many vectors as pairs
    lad = npp * s.lad * (0.5 if s.nq == 3 else 1.0)
    ladder = 2.0 * (0.5 * nh * lad * lad).sum()
    # rows (a,i) and columns (k,c) per conserved difference; of the channels that differ by the
    # flip of all spins one, of those without spin transfer a quarter of the products
    d = (st[A:, None] - st[None, :A]).reshape(-1, 5)
    kr, r = np.unique(s._key(d), return_counts=True)
    kc, c = np.unique(s._key(-d), return_counts=True)
    _, x, y = np.intersect1d(kr, kc, return_indices=True)
    r, c, slot = r[x].astype(float), c[y].astype(float), kr[x] % s.nq
    sz = slot - 1 if s.nq == 3 else slot // 3 - 1
    ph = 4.0 * (r * c * c * np.where(sz > 0, 1.0, np.where(sz == 0, 0.25, 0.0))).sum()
    return [float(u) for u in (s.n, ladder, (nh * nh * npp).sum(), ph, (lad * lad).sum(), (r * c * (sz >= 0)).sum())]


_KEPT = {}


def work(case):
    do = case["do"]
    if do == "grad":
        par = 2 * H * H + H * F + H
        return dict(bytes=4.0 * case["rows"] * (F + 1) + 8.0 * par, flops=6.0 * case["rows"] * par)
    N, Z, n2 = case["N"], case.get("Z"), case["n2max"]
    if (N, Z, n2) not in _KEPT:
        _KEPT[N, Z, n2] = _counts(N, Z, n2)
    n, ladder, hh, ph, vpp, nx = _KEPT[N, Z, n2]
    k = len(_mesh(case["mesh"])) if case.get("mesh") else case.get("batch", 1)
    if do == "create":  # the interaction of holes and particles, summed up; nothing large is read
        return dict(bytes=8.0 * k * n, flops=6.0 * k * n)
    if do == "predict":
        return dict(bytes=8.0 * k * n, flops=0.5 * k * n * 2 * (2 * H * H + H * F + H))
    if do == "mbpt3":
        return dict(bytes=8.0 * k * (vpp + 2 * n + nx), flops=k * (ladder + hh + 0.5 * ph))
    if do == "pp":
        return dict(bytes=8.0 * vpp + 16.0 * n, flops=2 * ladder)
    if do == "ph":
        return dict(bytes=16.0 * n + (8.0 if case["prec"] == "mixed" else 16.0) * nx, flops=ph)
    # a solve reads the interaction (pp and cross channels) and the amplitudes once per update
    updates = 122 if Z else (40 if case["tol_N"] < 1e-8 else 26 if case["tol_N"] < 1e-6 else 20)
    return dict(bytes=updates * k * ((8.0 if case["prec"] == "fp64" else 4.0) * (vpp + 2 * nx) + 16.0 * n),
                flops=updates * k * (ladder + 2 * hh + ph))
