"""FP64 products on the tensor cores (fp64_tc.cu): the right-hand side and its vector-Jacobian product against
the oracle at the sizes where the tiles, the K padding and the dispatch change, and the exact properties of
the digit form (power-of-two scaling, non-finite entries)."""
import numpy as np
import pytest

from oracle import g1g2_oracle as O

from .helpers import problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex128)).cuda()


def gpu_rhs(p, t, n, g2):
    dn, dg = torch.zeros_like(dev(n)), torch.zeros_like(dev(g2))
    p.rhs(t, dev(n), dev(g2), dn, dg)
    torch.cuda.synchronize()
    return dn.cpu().numpy(), dg.cpu().numpy()


# 16, 17: smallest sizes and K padded from odd; 32, 33: one and two column tiles; 48: 16-column padding of a tile
@pytest.mark.parametrize("nb,se,bosons", [(16, "SOA", False), (17, "GW", False), (21, "DSL", True), (24, "GWX", False),
                                          (25, "TPP", False), (31, "SOA", True), (32, "TPH", False), (33, "SOA", False),
                                          (48, "SOA", False)])
def test_rhs_matches_oracle(nb, se, bosons):
    """Two FP64 evaluations of sums of nb^3 (dn) and nb^2 (dG2) terms: each within a few hundred roundings of the
    exact sum, 1e-12 of the largest entry."""
    from paper_2002_12717_gb300.g1g2 import Propagator
    h, w, n, g2, D, drv = problem(nb, se, False, nb % 2 == 1, seed=300 + nb)
    prob = O.Problem(h, w, se, False, D, drv.f, bosons=bosons)
    want = O.rhs(prob, 0.7, n, g2)
    with Propagator(h, w, n, None, se, "fp64", bosons=bosons) as p:
        p.set_drive(D, drv)
        got = gpu_rhs(p, 0.7, n, g2)
    for a, b in zip(got, want):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()


def test_power_of_two_scaling_is_exact():
    """The commutator alone (w = 0): digits and exponents of 2^k G2 are those of G2, shifted."""
    from paper_2002_12717_gb300.g1g2 import Propagator
    nb = 24
    h, w, n, g2, D, drv = problem(nb, "SOA", False, False, seed=9)
    with Propagator(h, 0 * w, n, None, "SOA", "fp64") as p:
        _, ref = gpu_rhs(p, 0.0, n, g2)
        for k in (-700, 500):
            _, got = gpu_rhs(p, 0.0, n, np.ldexp(g2.real, k) + 1j * np.ldexp(g2.imag, k))
            assert np.array_equal(got.real, np.ldexp(ref.real, k)) and np.array_equal(got.imag, np.ldexp(ref.imag, k))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_entries_reach_the_same_outputs(bad):
    """A NaN or an Inf of G2 has no digits: every output that a plain sum takes it into is non-finite, no
    other is, and the others keep their values."""
    from paper_2002_12717_gb300.g1g2 import Propagator
    nb = 20
    h, w, n, g2, D, drv = problem(nb, "SOA", False, False, seed=11)
    with Propagator(h, w, n, None, "SOA", "fp64") as p:
        _, clean = gpu_rhs(p, 0.0, n, g2)
        g2 = g2.copy()
        g2[1, 2, 3, 4] = bad
        _, got = gpu_rhs(p, 0.0, n, g2)
    i, j, k, l = np.indices(g2.shape)
    hit = (((j == 2) & (k == 3) & (l == 4)) | ((i == 1) & (k == 3) & (l == 4)) | ((i == 1) & (j == 2) & (l == 4))
           | ((i == 1) & (j == 2) & (k == 3)))
    assert not np.isfinite(got[hit]).any()
    assert np.isfinite(got[~hit]).all()
    assert np.abs(got[~hit] - clean[~hit]).max() <= 1e-15 * np.abs(clean).max()


# around the lines between the CUDA-core and the digit products: pair products from nb = 12, mode products from nb = 19
# (their padded K and ragged tiles on both sides), split tiles of a pair product at nb = 27
@pytest.mark.parametrize("nb,se,bosons", [(5, "GW", False), (11, "GW", True), (12, "GWX", False), (13, "TPP", False),
                                          (14, "DSL", False), (15, "GW", False), (18, "SOA", True), (19, "SOA", False),
                                          (27, "GW", False)])
def test_rhs_matches_oracle_across_the_dispatch(nb, se, bosons):
    """As test_rhs_matches_oracle: 1e-12 of the largest entry."""
    test_rhs_matches_oracle(nb, se, bosons)


def test_results_near_the_end_of_the_exponent_range():
    """The commutator alone at 2^-1000 G2, where the conversion of the integer sums takes its careful path: the same
    numbers shifted, to the last subnormal bit (one rounding more there)."""
    from paper_2002_12717_gb300.g1g2 import Propagator
    nb, k = 24, -1000
    h, w, n, g2, D, drv = problem(nb, "SOA", False, False, seed=13)
    g2 = g2.copy()
    g2[2, 3] = 0.0                       # rows of zeros among them
    with Propagator(h, 0 * w, n, None, "SOA", "fp64") as p:
        _, ref = gpu_rhs(p, 0.0, n, g2)
        _, got = gpu_rhs(p, 0.0, n, np.ldexp(g2.real, k) + 1j * np.ldexp(g2.imag, k))
    for a, b in ((got.real, np.ldexp(ref.real, k)), (got.imag, np.ldexp(ref.imag, k))):
        assert np.abs(a - b).max() <= 16 * 2.0 ** -1074
