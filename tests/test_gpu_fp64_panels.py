"""Digit products beyond one tile of everything: vector-Jacobian products and gradients at sizes that use them (conjugated
operands, long contractions, digits of one matrix kept for the next product), and products cut into panels of rows,
columns and terms, which without a limit begin at nb = 65."""
import numpy as np
import pytest

from oracle import torch_oracle as TO
from paper_2002_12717_gb300 import inputs

from .helpers import problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex128)).cuda()


def reference(se, h, w, n, g, a, y):
    """Cotangents of (n, G2, h) by reverse-mode torch of the equations as sums."""
    e = torch.einsum
    h, w, n, g, a, y = (dev(x) for x in (h, w, n, g, a, y))
    h, n, g = (x.requires_grad_() for x in (h, n, g))
    wm = w - w.transpose(2, 3)
    nbar = torch.eye(h.shape[0], dtype=h.dtype, device="cuda") - n
    hhf = h + e("ikjl,lk->ij", wm, n)
    i = -1j * e("iklp,lpjk->ij", w, g)
    dn = -1j * (hhf @ n - n @ hhf) - (i + i.conj().T)
    c = (e("ip,pjkl->ijkl", hhf, g) + e("jq,iqkl->ijkl", hhf, g) - e("ijpl,pk->ijkl", g, hhf) - e("ijkp,pl->ijkl", g, hhf))
    x = e("pqrl,rk->pqkl", e("pqrs,sl->pqrl", w if se == "GW" else wm, n), n)
    x = e("ip,pjkl->ijkl", nbar, e("jq,pqkl->pjkl", nbar, x))
    if se in ("TPP", "DSL"):
        hc = (e("ip,pjkl->ijkl", nbar, e("jq,iqkl->ijkl", nbar, w)) - e("ip,pjkl->ijkl", n, e("jq,iqkl->ijkl", n, w)))
        x = x - e("ijpq,pqkl->ijkl", hc, g)
    if se in ("TPH", "DSL"):
        hc = e("ijkq,ql->ijkl", e("ip,pjkq->ijkq", n, w), nbar) - e("ijkq,ql->ijkl", e("ip,pjkq->ijkq", nbar, w), n)
        x = x - e("ipql,qjkp->ijkl", hc, g)
    c = c - x + x.permute(2, 3, 0, 1).conj()
    if se in ("GW", "DSL"):
        hc = e("ijkp,pl->ijkl", w, n) - e("jq,iqkl->ijkl", n, w)
        pi = e("qjpl,ipkq->ijkl", hc, g)
        c = c + pi - pi.permute(3, 2, 1, 0).conj()
    gh, gn, gg = torch.autograd.grad((dn, -1j * c), (h, n, g), (a, y))
    return [t.cpu().numpy() for t in (gn, gg, gh)]


def vjp(p, n, g, a, y):
    out = [torch.empty_like(dev(x)) for x in (n, g, n)]
    p.rhs_vjp(0.0, dev(n), dev(g), dev(a), dev(y), *out)
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in out]


# digits in pair products alone (12, 13), mode products too (19, 20), long contractions too (22, 24; two phases at 33)
@pytest.mark.parametrize("nb,se,complex_w", [(12, "GW", False), (13, "GW", True), (13, "TPP", False), (13, "DSL", True),
                                             (19, "SOA", True), (20, "TPH", False), (22, "TPP", True), (24, "SOA", True),
                                             (24, "GW", True), (24, "DSL", False), (33, "SOA", False)])
def test_vjp_matches_reverse_mode(nb, se, complex_w):
    """Sums of up to nb^3 terms in another order: 1e-12 of the largest entry."""
    from paper_2002_12717_gb300.g1g2 import Propagator
    h, w, n, g2, _, _ = problem(nb, se, False, complex_w, seed=nb, drive=False)
    rng = np.random.default_rng(nb)
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    a, y = z(nb, nb), z(*(nb,) * 4)
    with Propagator(h, w, n, None, se, "fp64", sym_tol=-1.0) as p:
        got = vjp(p, n, g2, a, y)
    for x, r in zip(got, reference(se, h, w, n, g2, a, y)):
        assert np.abs(x - r).max() <= 1e-12 * np.abs(r).max()


# KiB of digits per operand: a pair product needs 2304 for a tile at nb = 24 and 6400 at nb = 40, a long contraction 256 or 512 for
# a segment, a mode product 96 to 160 for a tile: each limit leaves several ragged panels of all of them
@pytest.mark.parametrize("nb,se,kib", [(24, "GW", 2400), (24, "GW", 5000), (24, "DSL", 2400), (27, "SOA", 600), (27, "SOA", 1300),
                                       (40, "TPP", 6500), (40, "TPP", 14000)])
def test_panels_agree_with_whole_products(nb, se, kib):
    """Mode and pair products form every element alike whatever the panels (dG2 to the last bit); panels of a long
    contraction change the order in which its segments are added (1e-13 of the largest entry, a few hundred roundings)."""
    from paper_2002_12717_gb300.g1g2 import OK, Propagator
    h, w, n, g2, _, _ = problem(nb, se, drive=False, seed=nb)
    rng = np.random.default_rng(nb)
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    a, y = z(nb, nb), z(*(nb,) * 4)

    def run(p):
        dn, dg = torch.empty_like(dev(n)), torch.empty_like(dev(g2))
        p.profile(True)
        p.rhs(0.0, dev(n), dev(g2), dn, dg)
        torch.cuda.synchronize()
        launches = {k: v[0] for k, v in p.profile_report().items()}
        return [dn.cpu().numpy(), dg.cpu().numpy()] + vjp(p, n, g2, a, y), launches

    with Propagator(h, w, n, None, se, "fp64") as p:
        whole, few = run(p)
        assert p._lib.g1g2_set_digit_panel(p._ctx, kib << 10) == OK
        cut, many = run(p)
    # what ran on digits still does, in more launches
    assert all(many.get(k) == few.get(k) for k in ("fp64_zgemm", "fp64_zgemm_splitk"))
    assert many["fp64_tc_digits"] > few["fp64_tc_digits"]
    assert np.array_equal(cut[1], whole[1])
    for x, r in zip(cut, whole):
        assert np.abs(x - r).max() <= 1e-13 * np.abs(r).max()


def test_adjoint_matches_reverse_mode():
    """Gradients of the double occupancy of a 4 x 3 cluster (nb = 24: digits in mode products and long contractions, sparse
    operands) against reverse-mode autograd of the oracle; its 8 right-hand sides and their transposes: 1e-10."""
    from paper_2002_12717_gb300.g1g2 import Propagator
    m, steps, dt = 5, 2, 0.02
    d = inputs.hubbard_2d_spin_orbital(4, 3, U=2.0, n_controls=m, ta=0.0, tb=steps * dt)
    vals = 0.3 * np.sin(np.arange(m) + 1.0)
    with Propagator(d["h"], d["w"], d["n0"], None, "SOA", "fp64") as p:
        p.set_drive(d["D"], inputs.PiecewiseLinear(vals, 0.0, steps * dt))
        J, drive, wscale, gh = p.adjoint(dt, steps, objective=0, n_drive_params=m)
    model = TO.TorchSOA(d["h"], d["w"], d["D"])
    c = torch.tensor(vals, requires_grad=True)
    s = torch.ones((), dtype=torch.float64, requires_grad=True)
    hx = torch.zeros((24, 24), dtype=torch.complex128, requires_grad=True)
    n, g = TO.propagate(model, torch.as_tensor(d["n0"], dtype=torch.complex128),
                        torch.zeros((24,) * 4, dtype=torch.complex128), dt, steps, c, 0.0, steps * dt, s, hx)
    J_ref = TO.mean_double_occupancy(n, g)
    gc, gs, g_h = torch.autograd.grad(J_ref, (c, s, hx))
    g_h = ((g_h + g_h.conj().T) / 2).numpy()
    assert abs(J - float(J_ref.detach())) <= 1e-13
    assert np.abs(drive - gc.numpy()).max() <= 1e-10 * max(np.abs(gc.numpy()).max(), 1e-3)
    assert abs(wscale - float(gs)) <= 1e-10 * abs(float(gs))
    assert np.abs(gh - g_h).max() <= 1e-10 * np.abs(g_h).max()
