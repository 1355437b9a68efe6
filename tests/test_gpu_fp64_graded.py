"""FP64 products of operands whose entries differ by many orders of magnitude: every real and imaginary part of a result
against exact rational sums, within the a-priori bound of FP64 multiply-adds, n 2^-53 sum |a| |b| over its own n terms
(not relative to the largest entry)."""
from fractions import Fraction as F

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex128)).cuda()


def rhs(h, w, n, g2, se="SOA"):
    from paper_2002_12717_gb300.g1g2 import Propagator
    with Propagator(h, w, n, None, se, "fp64", sym_tol=-1.0) as p:
        dn, dg = torch.zeros_like(dev(n)), torch.zeros_like(dev(g2))
        p.rhs(0.0, dev(n), dev(g2), dn, dg)
        torch.cuda.synchronize()
    return dn.cpu().numpy(), dg.cpu().numpy()


def exact_dot(a, b):
    """(re, im) of sum a b as rationals, and the sums of |terms| of either part."""
    re = im = F(0)
    for x, y in zip(a, b):
        xr, xi, yr, yi = F(float(x.real)), F(float(x.imag)), F(float(y.real)), F(float(y.imag))
        re += xr * yr - xi * yi
        im += xr * yi + xi * yr
    a, b = np.asarray(a), np.asarray(b)
    sr = np.abs(a.real) @ np.abs(b.real) + np.abs(a.imag) @ np.abs(b.imag)
    si = np.abs(a.real) @ np.abs(b.imag) + np.abs(a.imag) @ np.abs(b.real)
    return re, im, sr, si


def graded(kind, nb, rng):
    """Hermitian h, w and G2 (w, G2 as nb^2 x nb^2 matrices) of decaying, sparse or imaginary-graded entries."""
    i = np.arange(nb)
    d2 = np.abs(i[:, None] - i[None, :]).astype(float)
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    h, w, g = z(nb, nb), z(nb, nb, nb, nb), z(nb, nb, nb, nb)
    if kind == "decay":                 # a gapped system: exponentially small far from the diagonal
        h *= np.exp(-d2)
        f = np.exp(-d2[:, :, None, None] - d2[None, None] - d2[:, None, :, None] - d2[None, :, None, :])
        w, g = w * f, g * f
    elif kind == "core":                # one orbital with huge matrix elements that the others do not reach
        h *= 1e-3
        h[0, 0] = 1e9
        for x in (w, g):
            x[0], x[:, 0], x[:, :, 0], x[:, :, :, 0] = 0, 0, 0, 0
        w[0, 0, 0, 0] = 1e9
    elif kind == "nearly-real":         # imaginary parts far below the real ones
        h, w, g = (x.real + 1e-13j * x.imag for x in (h, w, g))
    elif kind == "blocks":              # two blocks and a weak, noise-like coupling
        b = (i < nb // 2).astype(float)
        weak = np.where(b[:, None] == b[None, :], 1.0, 1e-17)
        h *= weak
        f = weak[:, :, None, None] * weak[None, None] * weak[:, None, :, None]
        w, g = w * f, g * f
    h = (h + h.conj().T) / 2
    herm = lambda x: (x + x.transpose(2, 3, 0, 1).conj()) / 2  # noqa: E731
    return h, herm(w), herm(g)


KINDS = ["decay", "core", "nearly-real", "blocks"]


def entries(size, dims, rng, count):
    """Sampled index tuples: the smallest nonzero outputs, and others at random."""
    a = np.abs(size).reshape(-1)
    nz = np.flatnonzero(a)
    pick = list(nz[np.argsort(a[nz])[:count]]) + list(rng.integers(0, a.size, count))
    return [np.unravel_index(int(e), dims) for e in pick]


# mode products: tiles of 48 columns (all orders at once) and of 80 (two phases)
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("nb", [24, 40])
def test_mode_products(kind, nb):
    """w = 0: dG2 = -i [h2, G2], four mode products of 2 nb real terms each, added up."""
    rng = np.random.default_rng(nb)
    h, _, g = graded(kind, nb, rng)
    _, dg = rhs(h, np.zeros((nb,) * 4), np.eye(nb) / 2, g)
    for i, j, k, l in entries(dg, dg.shape, rng, 60):
        re = im = F(0)
        sr = si = 0.0
        for a, b, s in ((h[i], g[:, j, k, l], 1), (h[j], g[i, :, k, l], 1), (h[:, k], g[i, j, :, l], -1),
                        (h[:, l], g[i, j, k], -1)):
            r, m, x, y = exact_dot(a, b)
            re, im, sr, si = re + s * r, im + s * m, sr + x, si + y
        got = dg[i, j, k, l]            # -i (re + i im)
        assert abs(F(float(got.real)) - im) <= F((2 * nb + 4) * EPS) * F(si)
        assert abs(F(float(got.imag)) + re) <= F((2 * nb + 4) * EPS) * F(sr)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("nb", [16, 24])
def test_pair_products(kind, nb):
    """TPP at n = 0 and h = 0: dG2 = -i (w G2 - (w G2)^dag), nb^2 x nb^2 x nb^2 (two and five segments)."""
    rng = np.random.default_rng(nb)
    _, w, g = graded(kind, nb, rng)
    _, dg = rhs(np.zeros((nb, nb)), w, np.zeros((nb, nb)), g, "TPP")
    w2, g2, dg = w.reshape(nb * nb, -1), g.reshape(nb * nb, -1), dg.reshape(nb * nb, -1)
    for a, b in entries(dg, dg.shape, rng, 20):
        r1, i1, x1, y1 = exact_dot(w2[a], g2[:, b])
        r2, i2, x2, y2 = exact_dot(w2[b], g2[:, a])
        re, im = r1 - r2, i1 + i2
        got, tol = dg[a, b], F((2 * nb * nb + 4) * EPS)
        assert abs(F(float(got.real)) - im) <= tol * F(y1 + y2)
        assert abs(F(float(got.imag)) + re) <= tol * F(x1 + x2)


@pytest.mark.parametrize("kind", KINDS)
def test_long_contraction(kind):
    """n = 0 and h = 0: dn = -(I + I^dag), I_ij = -i sum_klp w_iklp G2_lpjk.  Segments of at most 256 terms, added up
    pairwise by unit: fewer than 512 roundings on the way of any term."""
    nb = 24
    rng = np.random.default_rng(3)
    _, w, g = graded(kind, nb, rng)
    dn, _ = rhs(np.zeros((nb, nb)), w, np.zeros((nb, nb)), g)
    wi = w.reshape(nb, -1)                                       # (k, l, p)
    gj = g.transpose(2, 3, 0, 1).reshape(nb, -1)                 # G2_lpjk as (j), (k, l, p)
    for i, j in entries(dn, dn.shape, rng, 4):
        r1, i1, x1, y1 = exact_dot(wi[i], gj[j])
        r2, i2, x2, y2 = exact_dot(wi[j], gj[i])
        # -(-i s1 + conj(-i s2)) = i s1 - i conj(s2)
        re, im = -i1 - i2, r1 - r2
        tol = F(512 * EPS)
        assert abs(F(float(dn[i, j].real)) - re) <= tol * F(y1 + y2)
        assert abs(F(float(dn[i, j].imag)) - im) <= tol * F(x1 + x2)


def from_digits(d):
    """sum d_s 256^-s as the nearest FP64 number from below in magnitude."""
    v = sum(F(x) / F(256) ** s for s, x in enumerate(d))
    m = int(v * F(2) ** 60)
    cut = max(0, abs(m).bit_length() - 53)
    return float(F((abs(m) >> cut) << cut) / F(2) ** 60) * (1 if m >= 0 else -1)


@pytest.mark.parametrize("digits", [(63, 127, 127, 127, 127, 127, 127, 127), (-63, -128, -128, -128, -128, -128, -128, -128),
                                    (33, -128, -128, -128, -128, -128, -128, 0), (1, 127, 127, 127, 127, 127, 127, 127),
                                    (-1, -128, -128, -128, -128, -128, -128, -128),
                                    (0, 31, -128, -128, -128, -128, -128, -128)])
@pytest.mark.parametrize("lead", [False, True])
def test_coherent_digits(digits, lead):
    """Constant w and G2 whose digits all have one sign and nearly their largest magnitude, the sums that exceed the integers
    of an FP32 accumulator first; lead: with one entry of 32 per row and segment that fixes the exponent.  I = nb^3 w G2."""
    nb = 24
    x = from_digits(digits)
    w, g = np.full((nb,) * 4, x), np.full((nb,) * 4, 1j * x)
    if lead:
        w[:, :, ::4, 3] = 32.0
        g[::4, 3, :, :] = 32.0j
    dn, _ = rhs(np.zeros((nb, nb)), w, np.zeros((nb, nb)), g)
    a, b = w.reshape(nb, -1)[0], g.transpose(2, 3, 0, 1).reshape(nb, -1)[0].imag
    s = sum(F(float(p)) * F(float(q)) for p, q in zip(a, b))     # I = -i (i s) = s; dn = -2 s
    size = F(float(np.abs(a) @ np.abs(b)))
    assert np.all(dn == dn[0, 0]) and abs(F(float(dn[0, 0].real)) + 2 * s) <= F(512 * EPS) * 2 * size


@pytest.mark.parametrize("kind", KINDS)
def test_long_contractions_with_conjugated_operands(kind):
    """Vector-Jacobian product at n = 0, w = 0 and no cotangent of dn: hbar = i (Y1 + Y2 - Y3 - Y4), the contractions of Y
    with conj(G2) over all indices but one; fewer than 512 roundings on the way of a term of each, four additions."""
    from paper_2002_12717_gb300.g1g2 import Propagator
    nb = 24
    rng = np.random.default_rng(7)
    h, y, g = graded(kind, nb, rng)
    zero = np.zeros((nb, nb))
    with Propagator(h, np.zeros((nb,) * 4), zero, None, "SOA", "fp64", sym_tol=-1.0) as p:
        out = [torch.empty_like(dev(x)) for x in (zero, g, zero)]
        p.rhs_vjp(0.0, dev(zero), dev(g), dev(zero), dev(y), *out)
        torch.cuda.synchronize()
    hbar = out[2].cpu().numpy()
    flat = lambda x, m: np.moveaxis(x, m, 0).reshape(nb, -1)  # noqa: E731
    for a, b in entries(hbar, hbar.shape, rng, 3):
        re = im = F(0)
        sr = si = 0.0
        for u, v, sign in ((flat(y, 0)[a], flat(g, 0)[b], 1), (flat(y, 1)[a], flat(g, 1)[b], 1),
                           (flat(y, 2)[b], flat(g, 2)[a], -1), (flat(y, 3)[b], flat(g, 3)[a], -1)):
            r, m, x, z = exact_dot(u, v.conj())
            re, im, sr, si = re + sign * r, im + sign * m, sr + x, si + z
        assert abs(F(float(hbar[a, b].real)) + im) <= F(516 * EPS) * F(si)       # i (re + i im)
        assert abs(F(float(hbar[a, b].imag)) - re) <= F(516 * EPS) * F(sr)
