"""Expired waits outside mw3_propagate, without a GPU fault.

With tc_wait_limit 0 the bounded mbarrier waits of the tile-major and of the FP64 angular step run out
at once (the other forms and the flush report one that did). The call that started the work has to say
so: after a wait that ran out its results come from tiles that were never written. An H_s application does not touch the propagation, which goes on as if nothing happened.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TIMEOUT = -6
# precision, n_gamma, states, tc_persist: FP64; tile-major, streamed, resident (by request and
# two states), without the parity split, one tile per CTA
FORMS = [("fp64", 24, 1, 4), ("fp64", 40, 2, 4), ("mixed", 24, 1, 4), ("mixed", 100, 1, 4),
         ("mixed", 24, 1, 2), ("mixed", 32, 2, 4), ("mixed", 24, 1, 1), ("mixed", 24, 1, 0)]


def _cfg(ng, ne):
    base = W.C3 if ne == 2 else W.C2
    return W.shrunk(base, "fail", NR=24, nr=20, ngamma=ng, J=[2], omega_max=2, nE=8, kmin=0,
                    vmax=-1, E_hi_eV=0.5, products=None)


def _expired(call):
    from paper_2412_10167_gb300 import mw3
    with pytest.raises(mw3.MW3Error) as e:
        call()
    assert e.value.code == TIMEOUT


@pytest.mark.parametrize("form", FORMS, ids=lambda f: "-".join(map(str, f)))
def test_expired_wait_of_an_hs_application_is_reported(form):
    from paper_2412_10167_gb300 import mw3
    precision, ng, ne, persist = form
    pr = mw3.Propagator(_cfg(ng, ne), precision=precision,
                        tuning=dict(tc_persist=persist) if precision == "mixed" else None)
    q = W.random_unit_state(pr.shape, 7)
    hs, (al, be) = pr.apply_hs(q), pr.lanczos(q, 4)
    pr.propagate(2)
    state = pr.state()[0].copy()
    pr.set_tuning("tc_wait_limit", 0)
    _expired(lambda: pr.apply_hs(q))
    _expired(lambda: pr.lanczos(q, 4))
    pr.set_tuning("tc_wait_limit", 1 << 22)
    assert np.array_equal(pr.apply_hs(q), hs)
    a2, b2 = pr.lanczos(q, 4)
    assert np.array_equal(a2, al) and np.array_equal(b2, be)
    assert np.array_equal(pr.state()[0], state)
    pr.propagate(2)
    pr.set_tuning("tc_wait_limit", 0)
    _expired(lambda: pr.propagate(2))
    pr.close()


def test_expired_wait_of_a_readers_flush_is_reported():
    from paper_2412_10167_gb300 import mw3
    pr = mw3.Propagator(_cfg(24, 1), precision="mixed")
    pr.propagate(20)                        # more pending iterations than are added on the fly
    pr.set_tuning("tc_wait_limit", 0)
    _expired(pr.probabilities)
    pr.close()
