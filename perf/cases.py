"""The calls that say how fast this framework is, over the range in which it is used.

A case is one public entry point at one size: `prepare` makes the problem and the context that a
program keeps, `run` is one pass, `exact` the same result from plain torch in 64 bits (the equations of
arXiv:2002.12717 written out as sums, without any code of this framework).

Sizes are those of the workloads in `inputs.py` and of the tests: the Hubbard chain and cluster, the
seeded general bases (w of rank 2 nb) at nb = 32, 48, 64, 96 under a pulse, and odd sizes between.  FP64 is the
default precision of a `Propagator`; bf16x4 is the tensor-core form that long runs of a real interaction take.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2002_12717_gb300 import inputs
from paper_2002_12717_gb300.g1g2 import Propagator, g1_rhs_noalloc

C128 = torch.complex128


def listed():
    return [
        # smallest: one propagation of the 8-site chain from host arrays to host arrays (launches and latency)
        dict(name="chain8-propagate", call="propagate", basis="chain", nb=8, selfenergy="SOA", precision="fp64",
             nsteps=25, obs_every=5),
        # a short run of the seeded basis in the default precision, energies recorded on the way
        dict(name="soa32-propagate", call="propagate", basis="general", nb=32, selfenergy="SOA", precision="fp64",
             nsteps=4, obs_every=2),
        # right-hand sides in FP64 (the callers' own integrators): odd size with a complex w, then the
        # pulse workloads
        dict(name="tpp27-complex", call="rhs", basis="general", nb=27, selfenergy="TPP", precision="fp64",
             complex_w=True),
        dict(name="gw48", call="rhs", basis="general", nb=48, selfenergy="GW", precision="fp64", complex_w=False),
        dict(name="soa64", call="rhs", basis="general", nb=64, selfenergy="SOA", precision="fp64", complex_w=False),
        # largest in FP64: the nb^6 polarisation at nb = 64
        dict(name="gw64", call="rhs", basis="general", nb=64, selfenergy="GW", precision="fp64", complex_w=False),
        # the tensor-core form: ladders and polarisation together at a ragged size, and the two headline workloads
        dict(name="dsl36-bf16x4", call="rhs", basis="general", nb=36, selfenergy="DSL", precision="bf16x4",
             complex_w=False),
        dict(name="gw64-bf16x4", call="rhs", basis="general", nb=64, selfenergy="GW", precision="bf16x4",
             complex_w=False),
        dict(name="soa96-bf16x4", call="rhs", basis="general", nb=96, selfenergy="SOA", precision="bf16x4",
             complex_w=False),
        # backward: one vector-Jacobian product (gradients through a caller's integrator), and the discrete
        # adjoint of the 4 x 4 cluster with its 64 controls
        dict(name="vjp-gw24", call="vjp", basis="general", nb=24, selfenergy="GW", precision="fp64", complex_w=False),
        dict(name="adjoint-4x4", call="adjoint", basis="cluster", nb=32, lx=4, ly=4, selfenergy="SOA",
             precision="fp64", nsteps=3, controls=64),
        # the memory-integral form, for comparisons with the time-local one
        dict(name="hfgkba-chain8", call="hfgkba", basis="chain", nb=8, selfenergy="SOA", precision="fp64", nsteps=100),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    call = rng.choice(["rhs", "rhs", "rhs", "bf16x4", "bf16x4", "propagate", "propagate", "vjp", "adjoint", "hfgkba",
                       "noalloc"])
    if call == "rhs":
        se = rng.choice(["SOA", "GW", "GWX", "TPP", "TPH", "DSL"])
        nb = _log_int(rng, 6, {"SOA": 72, "DSL": 48}.get(se, 60))
        return dict(call="rhs", basis="general", nb=nb, selfenergy=se, precision="fp64",
                    complex_w=rng.random() < 0.3)
    if call == "bf16x4":
        se = rng.choice(["SOA", "SOA", "GW", "GWX", "TPP", "TPH", "DSL"])
        return dict(call="rhs", basis="general", nb=4 * _log_int(rng, 2, 18), selfenergy=se, precision="bf16x4",
                    complex_w=False)
    if call == "propagate":
        if rng.random() < 0.5:
            return dict(call="propagate", basis="chain", nb=_log_int(rng, 4, 32), selfenergy=rng.choice(["SOA", "GW"]),
                        precision="fp64", nsteps=rng.randint(5, 40), obs_every=rng.randint(1, 5))
        return dict(call="propagate", basis="general", nb=_log_int(rng, 5, 40), selfenergy=rng.choice(["HF", "SOA", "GW"]),
                    precision="fp64", nsteps=rng.randint(1, 4), obs_every=rng.randint(1, 2))
    if call == "vjp":
        return dict(call="vjp", basis="general", nb=_log_int(rng, 5, 40), selfenergy=rng.choice(["SOA", "GW", "TPP"]),
                    precision="fp64", complex_w=rng.random() < 0.3)
    if call == "adjoint":
        lx, ly = rng.choice([(2, 2), (3, 2), (4, 2), (3, 3), (5, 2), (4, 3)])
        return dict(call="adjoint", basis="cluster", nb=2 * lx * ly, lx=lx, ly=ly, selfenergy="SOA", precision="fp64",
                    nsteps=rng.randint(2, 8), controls=rng.randint(4, 64))
    if call == "hfgkba":
        return dict(call="hfgkba", basis="chain", nb=_log_int(rng, 4, 13), selfenergy="SOA", precision="fp64",
                    nsteps=rng.randint(20, 120))
    return dict(call="noalloc", basis="general", nb=_log_int(rng, 6, 64), selfenergy="SOA", precision="fp64",
                complex_w=rng.random() < 0.5)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _herm(x):
    return (x + x.conj().T) / 2


def _problem(case, seed):
    """h, w, n, G2 as CUDA tensors, and D with its drive: everything from the seed."""
    nb, basis = case["nb"], case["basis"]
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (seed + 1) + nb)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    crand = lambda *s: torch.complex(rand(*s), rand(*s))  # noqa: E731
    dev = lambda a: torch.as_tensor(np.asarray(a), dtype=C128, device="cuda")  # noqa: E731
    p = dict(restricted=basis == "chain", D=None, drive=None, G2=None)
    if basis == "chain":
        u = 1.0 + 0.05 * float(rand(1)[0])
        d = inputs.hubbard_chain_restricted(nb, U=u, quench=2.0 + 0.1 * float(rand(1)[0]), quench_sites=(nb + 1) // 2)
        p.update(h=dev(d["h"]), w=torch.as_tensor(d["w"], device="cuda"), n=dev(d["n0"]))
        return p
    if basis == "cluster":
        d = inputs.hubbard_2d_spin_orbital(case["lx"], case["ly"], U=2.0 + 0.1 * float(rand(1)[0]),
                                           n_controls=case["controls"], ta=0.0, tb=0.01 * case["nsteps"])
        drive = inputs.PiecewiseLinear(0.1 * rand(case["controls"]).cpu().numpy(), 0.0, 0.01 * case["nsteps"])
        p.update(h=dev(d["h"]), w=torch.as_tensor(d["w"], device="cuda"), n=dev(d["n0"]), D=dev(d["D"]), drive=drive)
    else:
        cw = case.get("complex_w", False)
        h = _herm(crand(nb, nb)) / math.sqrt(nb)
        b = 0.1 * (crand(2 * nb, nb, nb) if cw else rand(2 * nb, nb, nb))
        fac = (b + b.transpose(1, 2).conj()) / 2
        flat = fac.reshape(2 * nb, nb * nb)
        w = (flat.T @ flat).reshape(nb, nb, nb, nb).permute(0, 2, 1, 3).contiguous()
        # occupations between a filled and an empty shell, in the eigenbasis of h
        e, v = torch.linalg.eigh(h + 0.1 * _herm(crand(nb, nb)) / math.sqrt(nb))
        occ = 1.0 / (1.0 + torch.exp(4.0 * (e - e.median())))
        D = torch.diag(rand(nb)).to(C128)
        p.update(h=h, w=w, n=_herm((v * occ) @ v.conj().T), D=D, drive=inputs.GaussSine())
    # a correlated state: Hermitian and exchange-symmetric, antisymmetric where the source is w^-
    x = 1e-2 * crand(nb, nb, nb, nb)
    if case["selfenergy"] != "GW":
        x = x - x.transpose(2, 3)
    x = x + x.permute(1, 0, 3, 2)
    p["G2"] = (x + x.permute(2, 3, 0, 1).conj()).contiguous()
    return p


def _host(x):
    return None if x is None else x.cpu().numpy()


T0 = 4.6          # inside the pulse of the general bases
DT = {"chain": 0.02, "cluster": 0.01, "general": 0.01}


def prepare(case, seed):
    torch.cuda.set_device(0)
    p = _problem(case, seed)
    nb, call = case["nb"], case["call"]
    s = dict(case=case, h=p["h"], n=p["n"], G2=p["G2"])
    if call == "noalloc":
        s.update(w=p["w"].to(C128).contiguous(), dn=torch.empty_like(p["n"]))
        return s
    # w is symmetric by construction: large problems leave out the host's check of nb^4 entries
    s["prop"] = Propagator(_host(p["h"]), _host(p["w"]), _host(p["n"]), None, case["selfenergy"], case["precision"],
                           restricted=p["restricted"], sym_tol=1e-10 if nb <= 48 else -1.0)
    if p["D"] is not None:
        s["prop"].set_drive(_host(p["D"]), p["drive"])
    if call in ("rhs", "vjp"):
        s.update(dn=torch.empty_like(p["n"]), dG=torch.empty_like(p["G2"]))
    if call == "vjp":
        a, y = _cotangents(case, seed)
        s.update(a=a, Y=y, hbar=torch.empty_like(p["n"]))
    if call in ("propagate", "adjoint"):
        s.update(n=_host(p["n"]), G2=_host(p["G2"]))
    if call == "hfgkba":
        s.update(n=_host(p["n"]))
    torch.cuda.synchronize()
    return s


def _cotangents(case, seed):
    nb = case["nb"]
    g = torch.Generator(device="cuda")
    g.manual_seed(7919 * (seed + 1) + nb)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    return torch.complex(rand(nb, nb), rand(nb, nb)), torch.complex(rand(*(nb,) * 4), rand(*(nb,) * 4))


def run(state):
    case = state["case"]
    call, dt = case["call"], DT[case["basis"]]
    if call == "noalloc":
        g1_rhs_noalloc(state["h"], state["w"], state["n"], state["G2"], state["dn"])
        return state["dn"]
    p = state["prop"]
    if call == "rhs":
        p.rhs(T0, state["n"], state["G2"], state["dn"], state["dG"])
        return state["dn"], state["dG"]
    if call == "vjp":
        p.rhs_vjp(T0, state["n"], state["G2"], state["a"], state["Y"], state["dn"], state["dG"], state["hbar"])
        return state["dn"], state["dG"], state["hbar"]
    p.set_state(0.0 if case["basis"] != "general" else T0, state["n"], state["G2"])
    if call == "propagate":
        obs, density = p.propagate(dt, case["nsteps"], case["obs_every"])
        _, n, G2 = p.get_state()
        return dict(energies=np.array([[o[k] for k in ENERGIES] for o in obs]), density=density, n=n, G2=G2)
    if call == "adjoint":
        J, drive, wscale, gh = p.adjoint(dt, case["nsteps"], objective=0, n_drive_params=case["controls"])
        return dict(J=J, drive=drive, wscale=wscale, h=gh)
    return p.propagate_hfgkba(dt, case["nsteps"])


ENERGIES = ("n_particles", "e_one", "e_hf", "e_corr", "e_total")


# ---------------------------------------------------------------------------
# What one pass cannot do without
# ---------------------------------------------------------------------------

def _rhs_cmacs(case):
    """Complex multiply-adds of one right-hand side as the equations have them."""
    nb, se = case["nb"], case["selfenergy"]
    if se == "HF":
        return nb ** 4
    if case["basis"] == "chain":            # on-site interaction, nearest neighbours
        return 30 * nb ** 4 * (2 if se == "GW" else 1)
    five = 9 + {"GW": 2, "GWX": 2, "TPP": 4, "TPH": 4, "DSL": 10}.get(se, 0)
    six = {"GW": 1, "GWX": 1, "TPP": 1, "TPH": 1, "DSL": 3}.get(se, 0)
    return five * nb ** 5 + six * nb ** 6 + nb ** 4


def work(case):
    nb, call = case["nb"], case["call"]
    n4 = float(nb) ** 4
    w = 16.0 if case.get("complex_w", False) else 8.0
    f = 8.0 * _rhs_cmacs(case)
    if call == "noalloc":
        return {"bytes": 32.0 * n4, "flops": 8.0 * (nb ** 5 + nb ** 4)}
    if call == "rhs":
        return {"bytes": (32.0 + w) * n4, "flops": f}
    if call == "vjp":
        return {"bytes": (48.0 + w) * n4, "flops": 2.5 * f}
    if call == "propagate":
        return {"bytes": (32.0 + w) * n4, "flops": 4.0 * f * case["nsteps"]}
    if call == "adjoint":
        return {"bytes": (32.0 + w) * n4, "flops": 4.0 * 4.5 * f * case["nsteps"]}
    # hfgkba: every evaluation sums over the whole history
    m = case["nsteps"]
    return {"bytes": 16.0 * n4 * m * (m + 3), "flops": 2.0 * 2.0 * n4 * m * (m + 3) + 8.0 * 12 * nb ** 5 * 2 * m}


# ---------------------------------------------------------------------------
# The same in 64 bits from plain torch
# ---------------------------------------------------------------------------

class _Exact:
    def __init__(self, case, p):
        self.se, self.restricted, self.nb = case["selfenergy"], p["restricted"], case["nb"]
        self.h, self.D, self.drive, self.w = p["h"], p["D"], p["drive"], p["w"].to(C128)
        self.hubbard_gw = self.restricted and self.se == "GW"

    def exch(self, w):
        return w if self.restricted else w - w.transpose(2, 3)

    def hhf(self, h, w, n):
        # w^-_ikjl n_lk
        return h + torch.einsum("ikjl,lk->ij", self.exch(w), n)

    def h_of_t(self, t):
        return self.h if self.D is None else self.h + self.drive.f(t) * self.D

    def ladder_hcorr(self, w, n):
        e = torch.einsum
        nbar = torch.eye(self.nb, dtype=C128, device=n.device) - n
        pp = e("ip,pjkl->ijkl", nbar, e("jq,iqkl->ijkl", nbar, w)) - e("ip,pjkl->ijkl", n, e("jq,iqkl->ijkl", n, w))
        ph = (e("ijkq,ql->ijkl", e("ip,pjkq->ijkq", n, w), nbar) - e("ijkq,ql->ijkl", e("ip,pjkq->ijkq", nbar, w), n))
        return pp, ph

    def source(self, w, n):
        """A = (nbar nbar) w (n n); the source term is -A + A^dag."""
        e = torch.einsum
        nbar = torch.eye(self.nb, dtype=C128, device=n.device) - n
        x = e("pqrs,sl->pqrl", w, n)
        x = e("pqrl,rk->pqkl", x, n)
        x = e("jq,pqkl->pjkl", nbar, x)
        return e("ip,pjkl->ijkl", nbar, x)

    def commutator(self, hhf, G):
        e = torch.einsum
        return (e("ip,pjkl->ijkl", hhf, G) + e("jq,iqkl->ijkl", hhf, G) - e("ijpl,pk->ijkl", G, hhf)
                - e("ijkp,pl->ijkl", G, hhf))

    def dn(self, hhf, n, I):
        return -1j * (hhf @ n - n @ hhf) - (I + I.conj().T)

    def rhs(self, h, w, n, G):
        e = torch.einsum
        hhf = self.hhf(h, w, n)
        if self.se == "HF":
            return self.dn(hhf, n, torch.zeros_like(n)), torch.zeros_like(G)
        I = -1j * e("iklp,lpjk->ij", w, G)
        r = self.commutator(hhf, G)
        A = self.source(w if self.restricted or self.se == "GW" else self.exch(w), n)
        if self.se in ("TPP", "DSL"):
            A = A - e("ijpq,pqkl->ijkl", self.ladder_hcorr(w, n)[0], G)
        if self.se in ("TPH", "DSL"):
            A = A - e("ipql,qjkp->ijkl", self.ladder_hcorr(w, n)[1], G)
        r = r - A + A.permute(2, 3, 0, 1).conj()
        if self.se in ("GW", "GWX", "DSL"):
            hc = e("ijkp,pl->ijkl", w, n) - e("jq,iqkl->ijkl", n, w)
            pi = e("qjpl,ipkq->ijkl", hc, G)
            r = r + pi - pi.permute(3, 2, 1, 0).conj()
        return self.dn(hhf, n, I), -1j * r

    def rhs_chain_gw(self, h, n, G, S):
        """Both spin blocks of the on-site problem: G opposite spins, S the same spin."""
        e = torch.einsum
        w = self.w
        u = torch.einsum("iiii->i", w)
        hhf = self.hhf(h, w, n)

        def pol(x):
            a = e("j,ijkj->ijk", u, x)       # sum over the site of the on-site interaction
            pi = e("jl,ijk->ijkl", n, a) - e("jl,ilk->ijkl", n, e("l,ilkl->ilk", u, x))
            return pi - pi.permute(3, 2, 1, 0).conj()

        A = self.source(w, n)
        dG = self.commutator(hhf, G) - A + A.permute(2, 3, 0, 1).conj() + pol(S)
        dS = self.commutator(hhf, S) + pol(G)
        return self.dn(hhf, n, -1j * e("iklp,lpjk->ij", w, G)), -1j * dG, -1j * dS

    def step(self, t, y, dt, h=None, w=None, drive=None):
        w = self.w if w is None else w

        def f(tt, z):
            ht = self.h_of_t(tt) if h is None else h + drive(tt) * self.D
            return self.rhs_chain_gw(ht, *z) if self.hubbard_gw else self.rhs(ht, w, *z)

        add = lambda a, c, b: tuple(x + c * k for x, k in zip(a, b))  # noqa: E731
        k1 = f(t, y)
        k2 = f(t + dt / 2, add(y, dt / 2, k1))
        k3 = f(t + dt / 2, add(y, dt / 2, k2))
        k4 = f(t + dt, add(y, dt, k3))
        return tuple(x + dt / 6 * (a + 2 * b + 2 * c + d) for x, a, b, c, d in zip(y, k1, k2, k3, k4))

    def energies(self, t, n, G):
        h, s = self.h_of_t(t), 2.0 if self.restricted else 1.0
        e1 = s * torch.einsum("ij,ji->", h, n).real
        ehf = 0.5 * s * torch.einsum("ij,ji->", self.hhf(h, self.w, n) - h, n).real
        ec = torch.zeros_like(e1) if self.se == "HF" else -0.5 * s * torch.einsum("ijkl,klij->", self.w, G).real
        return [float(x) for x in (s * torch.trace(n).real, e1, ehf, ec, e1 + ehf + ec)]


def exact(case, seed):
    p = _problem(case, seed)
    x = _Exact(case, p)
    call, dt, nb = case["call"], DT[case["basis"]], case["nb"]
    t0 = T0 if case["basis"] == "general" else 0.0
    n, G = p["n"], p["G2"]
    if G is None:
        G = torch.zeros((nb,) * 4, dtype=C128, device="cuda")
    if call == "noalloc":
        I = -1j * torch.einsum("iklp,lpjk->ij", x.w, G)
        return x.dn(x.hhf(p["h"], x.w, n), n, I)
    if call == "rhs":
        return x.rhs(x.h_of_t(T0), x.w, n, G)
    if call == "vjp":
        a, Y = _cotangents(case, seed)
        h, n, G = (v.clone().requires_grad_() for v in (x.h_of_t(T0), n, G))
        out = x.rhs(h, x.w, n, G)
        gh, gn, gG = torch.autograd.grad(out, (h, n, G), (a, Y))
        return gn, gG, gh
    if call == "propagate":
        y = (n, G) + ((torch.zeros_like(G),) if x.hubbard_gw else ())
        rec, dens, t, s = [], [], t0, 2.0 if x.restricted else 1.0
        for m in range(case["nsteps"] + 1):
            if m:
                y, t = x.step(t, y, dt), t + dt
            if m % case["obs_every"] == 0:
                rec.append(x.energies(t, y[0], y[1]))
                dens.append((s * torch.diagonal(y[0]).real).cpu().numpy())
        return dict(energies=np.array(rec), density=np.array(dens), n=y[0], G2=y[1])
    if call == "adjoint":
        return _exact_adjoint(case, x, n, G, dt)
    return _exact_hfgkba(case, x, n, dt)


def _exact_adjoint(case, x, n, G, dt):
    m, steps = case["controls"], case["nsteps"]
    theta = torch.tensor(x.drive.values, device="cuda").requires_grad_()
    scale = torch.ones((), dtype=torch.float64, device="cuda").requires_grad_()
    h = x.h.clone().requires_grad_()
    width = (x.drive.tb - x.drive.ta) / (m - 1)

    def f(t):
        u = (t - x.drive.ta) / width
        if u <= 0 or u >= m - 1:
            return theta[0 if u <= 0 else m - 1]
        k = min(int(math.floor(u)), m - 2)
        return (1 - (u - k)) * theta[k] + (u - k) * theta[k + 1]

    y, w = (n, G), x.w * scale
    for k in range(steps):
        y = x.step(k * dt, y, dt, h=h, w=w, drive=f)
    up = torch.arange(0, case["nb"], 2, device="cuda")
    dn = up + 1
    nn, g = y
    d = (nn[up, up] * nn[dn, dn] - nn[up, dn] * nn[dn, up]).real - g[up, dn, up, dn].real
    J = d.mean()
    gt, gs, gh = torch.autograd.grad(J, (theta, scale, h))
    return dict(J=float(J.detach()), drive=gt, wscale=float(gs), h=(gh + gh.conj().T) / 2)


def _exact_hfgkba(case, x, n, dt):
    e = torch.einsum
    nb, steps = case["nb"], case["nsteps"]
    wsrc = x.w if x.restricted else x.exch(x.w)

    def psi(n_):
        A = x.source(wsrc, n_)
        return -1j * (A.permute(2, 3, 0, 1).conj() - A)

    def memory(us, qs, u_now):
        if len(qs) == 1:
            return torch.zeros_like(qs[0])
        q = torch.stack(qs)
        v = e("ip,kjp->kij", u_now, torch.stack(us).conj())
        wt = torch.full((len(qs),), dt, dtype=torch.float64, device="cuda")
        wt[0] = wt[-1] = 0.5 * dt
        y = e("kjq,kiqrs->kijrs", v, e("kip,kpqrs->kiqrs", v, q))
        y = e("kijrl,kcr->kijcl", e("kijrs,kls->kijrl", y, v.conj()), v.conj())
        return e("k,kijcl->ijcl", wt.to(C128), y)

    def derivs(n_, u_, g_):
        hhf = x.hhf(x.h, x.w, n_)
        return x.dn(hhf, n_, -1j * e("iklp,lpjk->ij", x.w, g_)), -1j * hhf @ u_

    u = torch.eye(nb, dtype=C128, device="cuda")
    us, qs, out = [u], [psi(n)], [n]
    g = torch.zeros((nb,) * 4, dtype=C128, device="cuda")
    for _ in range(steps):
        dn1, du1 = derivs(n, u, g)
        np_, up_ = n + dt * dn1, u + dt * du1
        gp = memory(us + [up_], qs + [psi(np_)], up_)
        dn2, du2 = derivs(np_, up_, gp)
        n, u = n + dt / 2 * (dn1 + dn2), u + dt / 2 * (du1 + du2)
        us.append(u)
        qs.append(psi(n))
        g = memory(us, qs, u)
        out.append(n)
    return torch.stack(out)
