"""The bounded waits of the panel kernel and of the FP64 slice kernel, made to run out as in test_gpu_failure (copies
withheld by the host, a short limit): QCX_ERR_TIMEOUT, no eps, and the same context then gives the result of an
undisturbed call, bit for bit."""
import numpy as np
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED, qcx, states
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("route,prec,size", [("panels", QCX_MIXED, dict(n_k=6, nv=4, nc=12, ng=129, nw=120)),
                                             ("fp64_slices", QCX_FP64, dict(n_k=4, nv=2, nc=5, ng=65, nw=9))])
def test_wait_timeout_is_reported_and_the_context_recovers(route, prec, size):
    p = synth.make_tiny(nq=1, **size)
    p.w = synth.omega_grid(40.0, size["nw"])
    ctx = context()
    try:
        states.load_problem(ctx, p, [0])
        ctx.pair_density(0, p.G_int, prec)
        good = ctx.chi0(0, p.w, p.eta, prec, want=True)
        assert ctx.chi0_route(prec) == route
        ctx.set_wait_limit(200000)                  # ~0.1 ms of clock cycles
        ctx.set_fault_injection(True)
        for _ in range(2):
            with pytest.raises(qcx.QcxError) as e:
                ctx.chi0(0, p.w, p.eta, prec, want=True)
            assert e.value.status == 6              # QCX_ERR_TIMEOUT
            with pytest.raises(qcx.QcxError) as e:  # no eps was produced
                ctx.invert_eps(0, prec)
            assert e.value.status == 7
        ctx.set_fault_injection(False)
        ctx.set_wait_limit(4000000000)
        again = ctx.chi0(0, p.w, p.eta, prec, want=True)
        assert ctx.chi0_route(prec) == route
        ctx.invert_eps(0, prec)
    finally:
        ctx.close()
    assert np.array_equal(good, again)
