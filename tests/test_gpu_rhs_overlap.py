"""g1g2_rhs with dG2 written over (or across) the G2 it is evaluated at: the derivative is that of the call with
separate buffers, bit by bit, in the general basis and on the Hubbard path, whose stage kernel reads G2 at
other elements than it writes."""
import numpy as np
import pytest

from paper_2002_12717_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hubbard", [True, False])
@pytest.mark.parametrize("nb", [4, 12, 16])
@pytest.mark.parametrize("shift", [0, 1, 37])
def test_dg2_may_overlap_g2(hubbard, nb, shift):
    from paper_2002_12717_gb300.g1g2 import Propagator
    rng = np.random.default_rng(10 * nb + shift)
    h = inputs.grid_hopping(nb, 1, 1.0) + np.diag(rng.uniform(-0.5, 0.5, nb))
    w = inputs.onsite_w_restricted(nb, 2.0)
    n, g2 = inputs.random_state(nb, rng, soa=False)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex128)).cuda()  # noqa: E731
    nd, g, n4 = dev(n), dev(g2).reshape(-1), nb ** 4
    with Propagator(h, w, n, None, "SOA", "fp64", restricted=True) as p:
        p.hubbard_path = hubbard
        dn, dg, dn2 = torch.empty_like(nd), torch.empty_like(g), torch.empty_like(nd)
        p.rhs(0.0, nd, g, dn, dg)
        for _ in range(5):
            buf = torch.zeros(n4 + shift, dtype=torch.complex128, device="cuda")
            buf[:n4] = g
            p.rhs(0.0, nd, buf[:n4], dn2, buf[shift:])
            assert torch.equal(buf[shift:], dg) and torch.equal(dn2, dn)
