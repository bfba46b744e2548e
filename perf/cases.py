"""Performance cases of the library: single operators, solves, forces and
whole calls through the public Python binding, on the lattices of the run
files, the benchmark and the tests (4^3 .. 32^3 x 64, (T, X, Y, Z) order).

Inputs are synthetic: SU(3) links near the identity (the spread of
exp(i eps A), eps = 0.3), complex Gaussian spinors of density exp(-|eta|^2),
N(0, 1) momenta, all drawn on the GPU from the seed.  On these links the
hopping matrix is critical near kappa = 0.1325; kappa = 0.125 and 0.130 lie
below it, where a solve to 1e-12 takes 100 to 250 iterations (towards the
near-critical regime of the thermalised ensembles), and kappa = 0.156, 0.1575,
the production values, lie above it (about 50 iterations).

Outputs come in the device layouts of include/hmc.h, with the padding of a
field (sites are rounded up to 32) cleared once in prepare() or left out.
"""
import math

import numpy as np
import torch

from paper_1805_03560_gb300 import autograd as A
from paper_1805_03560_gb300 import hmc as H

DEV = "cuda"
EPS = 0.3
BETA = 5.6
PREC = {"f64": H.F64, "f32": H.F32, "f16": H.F16, "bf16": H.BF16, "f64e": H.F64E}


def _L(case):
    return (case["T"], case["X"], case["Y"], case["Z"])


def _volume(L):
    return L[0] * L[1] * L[2] * L[3]


# ---- the cases ----------------------------------------------------------------------


def listed():
    return [
        # one Mhat on the smallest lattice in use (differentiation, 8^3 x 16):
        # two launches of 4096 sites, latency and launch cost
        _case("mhat_f32_8x16", "mhat", (16, 8, 8, 8), prec="f32", n_rhs=1, kappa=0.156),
        # Mhat on the benchmark lattice, the operator of every solve
        _case("mhat_f32_24x48", "mhat", (48, 24, 24, 24), prec="f32", n_rhs=1, kappa=0.1575),
        # twelve right-hand sides in one launch (mass-preconditioned and
        # filter right-hand sides batched)
        _case("mhat_f32_rhs12_24x48", "mhat", (48, 24, 24, 24), prec="f32", n_rhs=12,
              kappa=0.1575),
        # a solve on a small lattice whose extents are no multiple of
        # anything (Vh = 8400, a ragged last block)
        _case("cg_f32_20x14x6x10", "cg", (20, 14, 6, 10), inner="f32", kappa=0.130),
        # the throughput configuration of the tests: 16^3 x 32, FP32 inner
        # precision, reliable updates in emulated FP64
        _case("cg_f32_16x32", "cg", (32, 16, 16, 16), inner="f32", kappa=0.130),
        # half storage of the inner solve on the benchmark lattice
        _case("cg_f16_24x48", "cg", (48, 24, 24, 24), inner="f16", kappa=0.1575),
        # the largest lattice in use, fields far above L2
        _case("cg_f32_32x64", "cg", (64, 32, 32, 32), inner="f32", kappa=0.130),
        # pseudo-fermion force of a molecular-dynamics step with the kappa^4
        # filter: Horner chains, two solves, ten outer-product pairs, all
        # FP64-accurate parts in emulated FP64 (the benchmark's force)
        _case("force_filter_24x48", "force", (48, 24, 24, 24), degree=9, solve=True,
              kappa=0.1575),
        # force of a rooted-polynomial pseudo-fermion (degree 16, no solve)
        _case("force_poly16_16x32", "force", (32, 16, 16, 16), degree=16, solve=False,
              kappa=0.130),
        # gauge force with the kappa^4 term, one per fine step
        _case("gauge_force_24x48", "gauge_force", (48, 24, 24, 24), kappa=0.1575),
        # a short trajectory of the kappa^4 leapfrog ensemble's lattice
        # (12^3 x 24): heatbath, actions, forces, link updates
        _case("trajectory_12x24", "trajectory", (24, 12, 12, 12), kappa=0.156, n_md=4),
        # gradient of the gauge and the pseudo-fermion action by autograd on
        # 8^3 x 16, everything in native FP64
        _case("autograd_8x16", "autograd", (16, 8, 8, 8), kappa=0.130),
    ]


def _case(name, kind, L, **kw):
    c = {"kind": kind, "T": L[0], "X": L[1], "Y": L[2], "Z": L[3], **kw}
    if name:
        c["name"] = name
    return c


def _draw_lattice(rng, v_min, v_max):
    """Even extents, volume spread over its logarithm."""
    while True:
        v = math.exp(rng.uniform(math.log(v_min), math.log(v_max)))
        s = (v / 2) ** 0.25
        L = [2 * max(2, round(s * rng.uniform(0.7, 1.4) / 2)) for _ in range(4)]
        L[0] = 2 * max(2, round(v / (L[1] * L[2] * L[3]) / 2))
        if L[0] <= 96 and v_min <= _volume(L) <= v_max:
            return tuple(L)


def draw(rng):
    kind = rng.choice(["mhat", "mhat", "cg", "cg", "force", "gauge_force", "trajectory",
                       "autograd"])
    if kind == "mhat":
        prec = rng.choice(["f32", "f32", "bf16", "f64"])
        n = rng.choice([1, 1, 2, 3, 4, 6, 8, 12]) if prec != "f64" else 1
        L = _draw_lattice(rng, 2048, 663552 if n > 1 else 2097152)
        return _case(None, kind, L, prec=prec, n_rhs=n,
                     kappa=rng.choice([0.150, 0.154, 0.156, 0.1575]))
    if kind == "cg":
        inner = rng.choice(["f32", "f32", "f16"])
        return _case(None, kind, _draw_lattice(rng, 4096, 1048576), inner=inner,
                     kappa=0.1575 if inner == "f16" else rng.choice([0.125, 0.130, 0.1575]))
    if kind == "force":
        solve = rng.random() < 0.5
        return _case(None, kind, _draw_lattice(rng, 8192, 663552), solve=solve,
                     degree=rng.choice([5, 6, 9, 15]) if solve else rng.choice([8, 16, 24]),
                     kappa=rng.choice([0.125, 0.130]))
    if kind == "gauge_force":
        return _case(None, kind, _draw_lattice(rng, 4096, 1048576), kappa=0.156)
    if kind == "trajectory":
        return _case(None, kind, _draw_lattice(rng, 4096, 65536), kappa=0.156,
                     n_md=rng.choice([2, 3, 4]))
    return _case(None, kind, _draw_lattice(rng, 4096, 32768), kappa=rng.choice([0.125, 0.130]))


# ---- inputs -------------------------------------------------------------------------


def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000 * int(seed) + stream)
    return g


def _normal(shape, seed, stream):
    return torch.randn(shape, dtype=torch.float64, device=DEV, generator=_gen(seed, stream))


def _links(L, seed):
    """SU(3) links [V, 4, 3, 3]: 1 + X + X^2/2 with X = i eps A, A = sum_a
    a_a lambda_a / 2, a_a ~ N(0, 1), rows orthonormalised."""
    V = _volume(L)
    out = torch.empty((V, 4, 3, 3), dtype=torch.complex128, device=DEV)
    flat = out.view(4 * V, 3, 3)
    a = _normal((4 * V, 8), seed, 1)
    for s in range(0, 4 * V, 1 << 20):
        X = 1j * EPS * _algebra(a[s:s + (1 << 20)])
        M = X + 0.5 * _mm(X, X)
        M = M + torch.eye(3, dtype=torch.complex128, device=DEV)
        r0 = M[:, 0] / M[:, 0].abs().square().sum(-1, keepdim=True).sqrt()
        r1 = M[:, 1] - (r0.conj() * M[:, 1]).sum(-1, keepdim=True) * r0
        r1 = r1 / r1.abs().square().sum(-1, keepdim=True).sqrt()
        flat[s:s + (1 << 20)] = torch.stack([r0, r1, torch.cross(r0, r1, dim=-1).conj()], 1)
    return out


def _algebra(a):
    """sum_a a_a lambda_a / 2 of components [..., 8]."""
    a = a.unbind(-1)
    d = a[7] / math.sqrt(3.0)
    z = torch.zeros_like(d)
    rows = [torch.complex(a[2] + d, z), torch.complex(a[0], -a[1]), torch.complex(a[3], -a[4]),
            torch.complex(a[0], a[1]), torch.complex(d - a[2], z), torch.complex(a[5], -a[6]),
            torch.complex(a[3], a[4]), torch.complex(a[5], a[6]), torch.complex(-2 * d, z)]
    m = 0.5 * torch.stack(rows, -1)
    return m.view(*m.shape[:-1], 3, 3)


def _gauss(L, seed, n=None):
    Vh = _volume(L) // 2
    shape = (Vh, 4, 3, 2) if n is None else (n, Vh, 4, 3, 2)
    return torch.view_as_complex(_normal(shape, seed, 2) * math.sqrt(0.5))


_ctx = []


def _context():
    """One library context per process, as a program keeps it."""
    if not _ctx:
        _ctx.append(H.Context(0))
    return _ctx[0]


def _clear(field):
    field.data.zero_()
    return field


def _filter(case):
    """Coefficients of a force: the kappa^4 filter truncated at the degree,
    or a polynomial of decaying coefficients (the rooted hierarchy's P_1)."""
    n = case["degree"]
    if case["solve"]:
        e = [1.0]
        for m in range(1, 200):
            e.append(-sum(e[m - j] for j in (1, 2) if j <= m) / m)
        b = [-sum(reversed(e[m + 1:])) for m in range(n + 1)]
        return np.array(b), math.exp(-1.5)
    # Taylor series of (1 - x)^(-1/2), the square root of the inverse
    b = [1.0]
    for m in range(1, n + 1):
        b.append(b[-1] * (m - 0.5) / m)
    return np.array(b), 0.0


SOLVER = {"reliable_delta": 1e-5, "f64_emul": 1}  # the production runner's defaults


def prepare(case, seed):
    L = _L(case)
    ctx = _context()
    kind = case["kind"]
    s = {"case": case, "L": L, "ctx": ctx}
    U = _links(L, seed)
    if kind == "mhat":
        p = PREC[case["prec"]]
        s["U"] = ctx.pack_gauge(L, U, p, H.LINK18 if case["prec"] == "f64" else H.LINK12)
        n = case["n_rhs"]
        s["in"] = ctx.pack_spinor(L, _gauss(L, seed, n if n > 1 else None), p)
        s["out"] = _clear(ctx.new_spinor(L, p, n))
    elif kind == "cg":
        p = PREC[case["inner"]]
        s["U"] = ctx.pack_gauge(L, U, H.F64, H.LINK18)
        s["Ulo"] = ctx.pack_gauge(L, U, p, H.LINK12)
        s["b"] = ctx.pack_spinor(L, _gauss(L, seed), H.F64)
        s["x"] = _clear(ctx.new_spinor(L, H.F64))
    elif kind == "force":
        s["U"] = ctx.pack_gauge(L, U, H.F64, H.LINK18)
        s["Ulo"] = ctx.pack_gauge(L, U, H.F32, H.LINK12)
        s["b"] = ctx.pack_spinor(L, _gauss(L, seed), H.F64)
        s["F"] = ctx.new_algebra(L)
        s["filter"] = _filter(case)
    elif kind == "gauge_force":
        s["U"] = ctx.pack_gauge(L, U, H.F64E, H.LINK18)
        s["F"] = ctx.new_algebra(L)
    elif kind == "trajectory":
        s["U"] = ctx.pack_gauge(L, U, H.F64, H.LINK18)
        s["P"] = ctx.pack_algebra(L, _normal((_volume(L), 4, 8), seed, 3))
        s["eta"] = ctx.pack_spinor(L, _gauss(L, seed), H.F64)
        s["U_end"], s["P_end"] = ctx.new_gauge(L, H.F64, H.LINK18), ctx.new_algebra(L)
        s["coeffs"] = H.filter_coeffs(2, 29)
    else:
        s["U"] = U.requires_grad_(True)
        s["phi"] = _gauss(L, seed)
    return s


# ---- one pass -----------------------------------------------------------------------


def _view(field, L):
    """A field's values in its storage type, without allocation padding."""
    S = _volume(L) // 2 * field.n_rhs
    d = field.data
    if field.prec == H.F64:
        return d[:S * 192].view(torch.float64)
    if field.prec == H.BF16:
        return d[:S * 48].view(torch.bfloat16)
    return d.view(torch.float32)


def run(s):
    case, L, ctx = s["case"], s["L"], s["ctx"]
    kind = case["kind"]
    if kind == "mhat":
        return _view(ctx.mhat(L, s["U"], s["out"], s["in"], case["kappa"]), L)
    if kind == "cg":
        # to the tolerance of the action solves
        ctx.cg_solve(L, s["U"], s["x"], s["b"], case["kappa"], 1e-12, U_lo=s["Ulo"],
                     inner_prec=PREC[case["inner"]], **SOLVER)
        return _view(s["x"], L)
    if kind == "force":
        b, alpha = s["filter"]
        s["F"].data.zero_()
        ctx.force_pf(L, s["U"], s["b"], case["kappa"], s["F"], tol=1e-12, U_lo=s["Ulo"],
                     inner_prec=H.F32, b=b, alpha=alpha, force_prec=H.F64E, **SOLVER)
        return s["F"].data
    if kind == "gauge_force":
        s["F"].data.zero_()
        ctx.force_hopexp(L, s["U"], BETA, case["kappa"], 2, F=s["F"], want_action=False)
        return s["F"].data
    if kind == "trajectory":
        # the run file's parameters, fewer steps of the same size; solves to
        # 1e-12 (the paper solves to machine precision)
        b, alpha, c = s["coeffs"]
        n = case["n_md"]
        r = ctx.trajectory(L, s["U"], s["P"], s["eta"], 1.0, beta=BETA, kappa=case["kappa"],
                           tau=math.sqrt(2.0) * n / 16, n_md=n, n_gauge=6, filter_k=2, n_t=15,
                           n_max=29, b=b, c=c, alpha=alpha, tol_md=1e-12, tol_action=1e-12,
                           inner_prec=H.F32, U_end=s["U_end"], P_end=s["P_end"],
                           force_prec=H.F64E, **SOLVER)
        return {"U": s["U_end"].data[:_volume(L) * 576].view(torch.float64),
                "P": s["P_end"].data, "H0": r["H0"], "H1": r["H1"], "plaq1": r["plaq1"]}
    S = A.gauge_action(ctx, L, s["U"], BETA, case["kappa"], 2)
    S = S + A.pf_action(ctx, L, s["U"], s["phi"], case["kappa"])
    (G,) = torch.autograd.grad(S, s["U"])
    return {"S": S.detach(), "G": G}


# ---- algorithmic work of one pass ----------------------------------------------------

_BYTES = {"f64": 8, "f64e": 8, "f32": 4, "f16": 2, "bf16": 2}
_HOP = 1320  # flops of a hemi-Dslash per output site


def _iterations(kappa):
    """Iterations of a solve to 1e-12 on these links (measured, rounded)."""
    return {0.125: 110, 0.130: 180}.get(kappa, 52)


def work(case):
    V = _volume(_L(case))
    Vh = V // 2
    kind, kappa = case["kind"], case["kappa"]
    if kind == "mhat":
        b = _BYTES[case["prec"]]
        R = 18 if case["prec"] == "f64" else 12
        n = case["n_rhs"]
        return {"bytes": 8 * Vh * R * b + 2 * 24 * Vh * n * b, "flops": (2 * _HOP + 48) * Vh * n}
    if kind == "cg":
        # per iteration every link once and x, r, p read and written once
        b = _BYTES[case["inner"]]
        it = _iterations(kappa)
        return {"bytes": it * Vh * (8 * 12 * b + 24 * (4 * b + 2 * 4)),
                "flops": it * Vh * (4 * _HOP + 300)}
    if kind == "force":
        n = case["degree"]
        hops = 2 * n + 2 * (n - 1) + 2 * n + (8 if case["solve"] else 0)
        by = 8 * Vh * 18 * 8 + 24 * Vh * 8 + 64 * Vh * 8
        fl = Vh * (hops * _HOP + 8 * n * 36 * 8)
        if case["solve"]:
            it = 2 * _iterations(kappa)
            by += it * Vh * (8 * 12 * 4 + 24 * (4 * 4 + 2 * 4))
            fl += it * Vh * (4 * _HOP + 300)
        return {"bytes": by, "flops": fl}
    if kind == "gauge_force":
        return {"bytes": 8 * Vh * 18 * 8 + 64 * Vh * 8, "flops": 8 * Vh * 13 * 216}
    if kind == "trajectory":
        n = case["n_md"]
        it = (2 * (n + 1) + 2) * _iterations(kappa)
        hops = (n + 1) * 98 + 200
        steps = 6 * n
        return {"bytes": it * Vh * (8 * 12 * 4 + 24 * (4 * 4 + 2 * 4))
                + steps * Vh * (2 * 8 * 18 * 8 + 3 * 64 * 8),
                "flops": it * Vh * (4 * _HOP + 300) + hops * Vh * _HOP
                + steps * 8 * Vh * 20 * 216}
    it = 2 * _iterations(kappa)
    return {"bytes": 2 * 8 * Vh * 18 * 8 + it * Vh * (8 * 18 * 8 + 24 * 6 * 8),
            "flops": it * Vh * (4 * _HOP + 300) + 8 * Vh * 13 * 216}


# ---- the same in 64 bits by plain torch ----------------------------------------------


def _mm(a, b):
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _dag(a):
    return a.conj().transpose(-1, -2)


class _Wilson:
    """Even/odd hopping matrix of the canonical links: chiral gamma basis,
    antiperiodic in time."""

    def __init__(self, L, U):
        self.L = L
        V = _volume(L)
        lex = torch.arange(V, device=DEV)
        x = torch.stack([lex // (L[1] * L[2] * L[3]), lex // (L[2] * L[3]) % L[1],
                         lex // L[3] % L[2], lex % L[3]])
        par = x.sum(0) % 2
        # lex of the h-th site of each parity
        self.site = [torch.empty(V // 2, dtype=torch.long, device=DEV) for _ in range(2)]
        for p in range(2):
            at = lex[par == p]
            self.site[p][at >> 1] = at
        st = [L[1] * L[2] * L[3], L[2] * L[3], L[3], 1]
        self.fwd, self.bwd, self.sf, self.sb = [], [], [], []
        for p in range(2):
            s, c = self.site[p], x[:, self.site[p]]
            self.fwd.append([s + torch.where(c[m] == L[m] - 1, 1 - L[m], 1) * st[m]
                             for m in range(4)])
            self.bwd.append([s + torch.where(c[m] == 0, L[m] - 1, -1) * st[m] for m in range(4)])
            one = torch.ones(V // 2, dtype=torch.float64, device=DEV)
            self.sf.append(torch.where(c[0] == L[0] - 1, -one, one))
            self.sb.append(torch.where(c[0] == 0, -one, one))
        self.U = U

    @staticmethod
    def gamma(mu, q):
        """gamma_mu psi; gamma_mu = [[0, B], [B^dag, 0]], B_0 = 1, B_k = -i sigma_k."""
        u0, u1, d0, d1 = q.unbind(-2)
        if mu == 0:
            r = (d0, d1, u0, u1)
        elif mu == 1:
            r = (-1j * d1, -1j * d0, 1j * u1, 1j * u0)
        elif mu == 2:
            r = (-d1, d0, u1, -u0)
        else:
            r = (-1j * d0, 1j * d1, 1j * u0, -1j * u1)
        return torch.stack(r, -2)

    def proj(self, mu, s, q):
        """(1 - s gamma_mu) q."""
        return q - s * self.gamma(mu, q)

    def hop(self, p, psi, dagger=False):
        """H_{p,1-p} psi (its gamma_5 conjugate with dagger)."""
        s = -1 if dagger else 1
        out = torch.zeros_like(psi)
        for mu in range(4):
            f, b = self.fwd[p][mu], self.bwd[p][mu]
            q = self.proj(mu, s, psi[f >> 1])
            U = self.U[self.site[p], mu]
            w = (U[:, None] * q[:, :, None, :]).sum(-1)
            out += self.sf[p][:, None, None] * w if mu == 0 else w
            q = self.proj(mu, -s, psi[b >> 1])
            U = _dag(self.U[b, mu])
            w = (U[:, None] * q[:, :, None, :]).sum(-1)
            out += self.sb[p][:, None, None] * w if mu == 0 else w
        return out

    def K(self, kappa, psi, dagger=False):
        return kappa * kappa * self.hop(0, self.hop(1, psi, dagger), dagger)

    def mhat(self, kappa, psi, dagger=False):
        return psi - self.K(kappa, psi, dagger)

    def solve(self, kappa, b):
        """(Mhat^dag Mhat)^-1 b by CG with the residual recomputed."""
        x, r = torch.zeros_like(b), b.clone()
        b2 = b.abs().square().sum()
        for _ in range(3):
            p, rr = r.clone(), r.abs().square().sum()
            stop = rr * 1e-22
            for _ in range(2000):
                if rr <= stop or rr <= 1e-31 * b2:
                    break
                q = self.mhat(kappa, self.mhat(kappa, p), True)
                a = rr / (p.conj() * q).real.sum()
                x, r = x + a * p, r - a * q
                new = r.abs().square().sum()
                p, rr = r + (new / rr) * p, new
            r = b - self.mhat(kappa, self.mhat(kappa, x), True)
            if r.abs().square().sum() <= 1e-29 * b2:
                break
        return x

    def pair_force(self, kappa, F, pairs):
        """F (canonical [V, 4, 8]) += the link derivative of
        2 kappa^2 Re sum W^dag H V, W = (A, H_eo^dag A), V = (B, H_oe B)."""
        k2 = kappa * kappa
        Q = {}
        for Ae, Be in pairs:
            W = [Ae, self.hop(1, Ae, True)]
            X = [Be, self.hop(1, Be)]
            for p in range(2):
                for mu in range(4):
                    n = self.fwd[p][mu] >> 1
                    a = self.proj(mu, 1, W[p])
                    b = self.proj(mu, -1, W[1 - p][n])
                    O1 = (X[1 - p][n][:, :, :, None] * a.conj()[:, :, None, :]).sum(1)
                    O2 = (X[p][:, :, :, None] * b.conj()[:, :, None, :]).sum(1)
                    U = self.U[self.site[p], mu]
                    q = _mm(U, O1) - _mm(O2, _dag(U))
                    if mu == 0:
                        q = self.sf[p][:, None, None] * q
                    Q[p, mu] = Q[p, mu] + q if (p, mu) in Q else q
        for (p, mu), q in Q.items():
            F[self.site[p], mu] -= k2 * _im_tr(q)

    def pf_force(self, kappa, phi, b, alpha):
        """Filtered action |(alpha Mhat^-1 + sum_n b_n K^n) phi|^2 (plain
        phi^dag (Mhat^dag Mhat)^-1 phi when b is None)."""
        F = torch.zeros((_volume(self.L), 4, 8), dtype=torch.float64, device=DEV)
        if b is None:
            x = self.solve(kappa, phi)
            self.pair_force(kappa, F, [(self.mhat(kappa, x), x)])
            return F
        Y = [b[-1] * phi]
        for c in reversed(b[:-1]):
            Y.append(c * phi + self.K(kappa, Y[-1]))
        Y.reverse()
        x1, pairs = Y[0], []
        if alpha:
            yt = alpha * self.solve(kappa, self.mhat(kappa, phi, True))
            x1 = x1 + yt
            pairs.append((self.mhat(kappa, self.solve(kappa, x1)), yt))
        xi = x1
        for i in range(1, len(b)):
            pairs.append((xi, Y[i]))
            xi = self.K(kappa, xi, True)
        self.pair_force(kappa, F, pairs)
        return F

    def gauge(self, beta):
        """(sum of Re Tr U_p, force of the plaquette action, canonical)."""
        L = self.L
        U = self.U.view(*L, 4, 3, 3)
        F = torch.empty((*L, 4, 8), dtype=torch.float64, device=DEV)
        plaq = 0.0
        for mu in range(4):
            Am = 0
            for nu in range(4):
                if nu == mu:
                    continue
                Um, Un = U[..., mu, :, :], U[..., nu, :, :]
                up = _mm(_mm(torch.roll(Un, -1, mu), _dag(torch.roll(Um, -1, nu))), _dag(Un))
                lo = _mm(_dag(_mm(Um, torch.roll(Un, -1, mu))), Un)
                Am = Am + up + torch.roll(lo, 1, nu)
                if nu > mu:
                    t = (Um * up.transpose(-1, -2)).sum((-1, -2)).real
                    plaq = plaq + t.sum()
            F[..., mu, :] = beta / 6.0 * _im_tr(_mm(U[..., mu, :, :], Am))
        return plaq, F.view(-1, 4, 8)


def _im_tr(q):
    """Im Tr(lambda_a q), a last."""
    r3 = 1.0 / math.sqrt(3.0)
    return torch.stack([
        q[..., 1, 0].imag + q[..., 0, 1].imag, q[..., 0, 1].real - q[..., 1, 0].real,
        q[..., 0, 0].imag - q[..., 1, 1].imag, q[..., 2, 0].imag + q[..., 0, 2].imag,
        q[..., 0, 2].real - q[..., 2, 0].real, q[..., 2, 1].imag + q[..., 1, 2].imag,
        q[..., 1, 2].real - q[..., 2, 1].real,
        (q[..., 0, 0].imag + q[..., 1, 1].imag - 2 * q[..., 2, 2].imag) * r3], -1)


def _beta_eff(case):
    return BETA + 96.0 * case["kappa"] ** 4


def _device_spinor(q, prec):
    """[n, Vh, 4, 3] in the device layout (values in 64 bits)."""
    n, Vh = q.shape[:2]
    e = torch.view_as_real(q.reshape(n, Vh, 12)).permute(1, 0, 2, 3).reshape(Vh * n, 24)
    if prec == "f32":
        pad = -(-e.shape[0] // 32) * 32
        f = torch.zeros((pad, 24), dtype=torch.float64, device=DEV)
        f[:e.shape[0]] = e
        return f.view(-1, 32, 6, 4).permute(0, 2, 1, 3).reshape(-1)
    per = 8 if prec == "bf16" else 2
    return e.view(-1, 24 // per, per).permute(1, 0, 2).reshape(-1)


def _device_algebra(W, F):
    return torch.stack([F[W.site[p]] for p in range(2)]).permute(0, 2, 3, 1).reshape(-1)


def exact(case, seed):
    L, kind, kappa = _L(case), case["kind"], case["kappa"]
    if kind == "trajectory":
        return None  # dozens of solves
    if any(v == 4 for v in L) and kind in ("gauge_force", "autograd"):
        return None  # straight lines around an extent of 4 enter the kappa^4 term
    U = _links(L, seed)
    W = _Wilson(L, U)
    if kind == "mhat":
        n = case["n_rhs"]
        q = _gauss(L, seed, n if n > 1 else None).view(n, -1, 4, 3)
        return _device_spinor(torch.stack([W.mhat(kappa, v) for v in q]), case["prec"])
    if kind == "cg":
        return _device_spinor(W.solve(kappa, _gauss(L, seed))[None], "f64")
    if kind == "force":
        return _device_algebra(W, W.pf_force(kappa, _gauss(L, seed), *_filter(case)))
    if kind == "gauge_force":
        return _device_algebra(W, W.gauge(_beta_eff(case))[1])
    plaq, F = W.gauge(_beta_eff(case))
    phi = _gauss(L, seed)
    S = -_beta_eff(case) / 3.0 * plaq + (phi.conj() * W.solve(kappa, phi)).real.sum()
    F = F + W.pf_force(kappa, phi, None, 0.0)
    return {"S": S, "G": 2.0 * _mm(1j * _algebra(F), U)}
