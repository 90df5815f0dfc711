"""FP64 pair densities and chi0 with device outputs do not wait for their kernels: both return while the context's stream is
still held by an earlier kernel; a wait of the slice kernel that gave up is reported by the inverse, and chi0 is NaN until
then.

The stream is held for ~0.4 s by torch's spin kernel (a fixed number of clock cycles); the calls must be back in half of that."""
import time

import pytest
import torch

import synth
from paper_2603_12326_gb300 import QCX_FP64, build, qcx, states

pytestmark = pytest.mark.gpu


@pytest.fixture()
def held():
    build.build()
    stream = torch.cuda.Stream()
    ctx = qcx.Context(0, stream=stream.cuda_stream)
    p = synth.make_tiny(n_k=4, nv=2, nc=5, ng=33, nq=1, nw=9)
    states.load_problem(ctx, p, [0])
    out = torch.zeros((9, 33, 33), dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    ctx.pair_density(0, p.G_int, QCX_FP64)               # buffers and kernels are there from here on
    ctx.chi0(0, p.w, p.eta, QCX_FP64, out=out)
    assert ctx.chi0_route(QCX_FP64) == "fp64_slices"
    ctx.sync()
    yield ctx, p, stream, out
    ctx.close()


def test_calls_return_before_their_kernels(held):
    ctx, p, stream, out = held
    want = out.clone()
    out.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        torch.cuda._sleep(800000000)
    t = time.perf_counter()
    ctx.pair_density(0, p.G_int, QCX_FP64)
    ctx.chi0(0, p.w, p.eta, QCX_FP64, out=out)
    t = time.perf_counter() - t
    assert not stream.query() and t < 0.2
    ctx.invert_eps(0, QCX_FP64)
    assert torch.equal(out, want)


def test_timeout_is_reported_by_the_inverse(held):
    ctx, p, stream, out = held
    ctx.set_wait_limit(200000)
    ctx.set_fault_injection(True)
    ctx.chi0(0, p.w, p.eta, QCX_FP64, out=out)
    with pytest.raises(qcx.QcxError) as e:
        ctx.invert_eps(0, QCX_FP64)
    assert e.value.status == 6                           # QCX_ERR_TIMEOUT
    assert bool(torch.isnan(out.real).all())
    with pytest.raises(qcx.QcxError) as e:               # no loss tables, no eps
        ctx.loss_function(0, QCX_FP64)
    assert e.value.status == 7
    with pytest.raises(qcx.QcxError) as e:
        ctx.invert_eps(0, QCX_FP64)
    assert e.value.status == 7
    ctx.set_fault_injection(False)
    ctx.set_wait_limit(4000000000)
    ctx.chi0(0, p.w, p.eta, QCX_FP64, out=out)
    ctx.invert_eps(0, QCX_FP64)
    assert bool(torch.isfinite(out.real).all())
