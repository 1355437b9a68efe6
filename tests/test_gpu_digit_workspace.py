"""The digit workspace of the FP64 products is optional: it is made after everything that a context needs, its absence
changes no result beyond rounding, and a context on the Hubbard path has none before it forms such products."""
import numpy as np
import pytest

from paper_2002_12717_gb300 import inputs

from .helpers import problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
MB = 1 << 20


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.complex128)).cuda()


def free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def rhs(p, n, g2):
    nd, gd = dev(n), dev(g2)
    dn, dg = torch.zeros_like(nd), torch.zeros_like(gd)
    p.rhs(0.0, nd, gd, dn, dg)
    torch.cuda.synchronize()
    return dn.cpu().numpy(), dg.cpu().numpy(), set(p.profile_report())


def test_init_needs_no_room_for_it():
    """GW at nb = 40: 14 tensors of 41 MB and a workspace of about 450 MB.  With 300 MB less than all of it free, init
    succeeds and the products run on the CUDA cores."""
    from paper_2002_12717_gb300.g1g2 import Propagator
    nb = 40
    h, w, n, g2, _, _ = problem(nb, "GW", drive=False, seed=nb)

    def run():
        with Propagator(h, w, n, None, "GW", "fp64", sym_tol=-1.0) as p:
            used = before - free()
            p.profile(True)
            return rhs(p, n, g2) + (used,)

    rhs_buffers = [dev(g2) for _ in range(4)]                # room for the call's own tensors in torch's pool
    before = free()
    a = run()
    assert any(k.startswith("fp64_tc") for k in a[2])
    del rhs_buffers
    keep = a[3] - 300 * MB + 4 * 16 * nb ** 4
    fill = torch.empty(free() - keep, dtype=torch.uint8, device="cuda")
    try:
        before = free()
        b = run()
    finally:
        del fill
        torch.cuda.empty_cache()
    assert not any(k.startswith("fp64_tc") for k in b[2])
    for x, y in zip(a[:2], b[:2]):
        assert np.abs(x - y).max() <= 1e-12 * np.abs(x).max()


def test_hubbard_context_makes_it_when_it_is_needed():
    from paper_2002_12717_gb300.g1g2 import Propagator
    nb = 24
    rng = np.random.default_rng(0)
    h, w = inputs.grid_hopping(nb, 1, 1.0), inputs.onsite_w_restricted(nb, 1.5)
    n, g2 = inputs.random_state(nb, rng, soa=False)
    with Propagator(h, w, n, None, "SOA", "fp64", restricted=True) as p:
        p.profile(True)
        _, a, kernels = rhs(p, n, g2)
        assert not any(k.startswith("fp64_tc") for k in kernels)
        before = free()
        p.hubbard_path = False
        assert before - free() > 10 * MB
        p.profile(True)
        _, b, kernels = rhs(p, n, g2)
        assert any(k.startswith("fp64_tc") for k in kernels)
    assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max()
