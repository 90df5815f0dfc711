"""qcx_rate with a loss table in page-locked host memory that an earlier copy on the context's stream is still to fill: its
inputs are taken in the stream's order.  The stream is held for ~0.2 s before that copy (torch's spin kernel)."""
import numpy as np
import pytest
import torch

from paper_2603_12326_gb300 import build, halo_params, qcx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,nw", [(40, 30), (700, 300)])        # below and above the size that is sent in one copy
def test_inputs_in_stream_order(nq, nw):
    build.build()
    stream = torch.cuda.Stream()
    ctx = qcx.Context(0, stream=stream.cuda_stream)
    try:
        q, w = np.linspace(0.1, 8.0, nq), np.linspace(0.05, 1.0, nw)
        L = torch.rand((nq, nw), dtype=torch.float64, device="cuda")
        host = torch.zeros((nq, nw), dtype=torch.float64).pin_memory()
        want = ctx.rate(q, w, L.cpu().numpy(), halo_params(), nQ=5)
        with torch.cuda.stream(stream):
            torch.cuda._sleep(400000000)
            host.copy_(L, non_blocking=True)
        got = ctx.rate(q, w, host, halo_params(), nQ=5)
    finally:
        ctx.close()
    assert np.any(want[0] > 0)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
