"""A kernel that gave up on a bounded wait is reported by the first call that synchronises, once, whatever queued it:
the error word is set from the host, as such a kernel sets it."""
import numpy as np
import pytest

from .helpers import problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("se,nb,precision", [("GW", 16, "fp64"), ("SOA", 24, "fp64"), ("SOA", 16, "bf16x4")])
@pytest.mark.parametrize("check", ["get_state", "synchronize", "observables"])
def test_timeout_is_reported_once(se, nb, precision, check):
    from paper_2002_12717_gb300.g1g2 import ETIMEOUT, OK, G1G2Error, Propagator
    h, w, n, g2, _, _ = problem(nb, se, drive=False, seed=nb)
    call = dict(get_state=lambda p: p.get_state(), synchronize=lambda p: p.synchronize(),
                observables=lambda p: p.observables())[check]
    with Propagator(h, w, n, g2, se, precision) as p:
        assert p._lib.g1g2_wait_inject(p._ctx) == OK
        with pytest.raises(G1G2Error) as e:
            call(p)
        assert e.value.code == ETIMEOUT
        p.set_state(0.0, n, g2)
        p.step(1e-3)
        p.synchronize()
        a = p.get_state()
        p.set_state(0.0, n, g2)
        p.step(1e-3)
        b = p.get_state()
        assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])


def test_context_without_bounded_waits():
    from paper_2002_12717_gb300.g1g2 import EUNSUPPORTED, Propagator
    h, w, n, g2, _, _ = problem(4, "SOA", drive=False)
    with Propagator(h, w, n, g2, "SOA", "fp64") as p:
        assert p._lib.g1g2_wait_inject(p._ctx) == EUNSUPPORTED
        p.synchronize()
