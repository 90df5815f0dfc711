"""What qcx_batch_info reports of a plan against what the profiler sees of one replay: the number of kernels, and the LU grid
that only the FP64 plan launches."""
import numpy as np
import pytest
import torch

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED, states
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [QCX_FP64, QCX_MIXED])
def test_kernels_per_replay(prec):
    from torch.profiler import ProfilerActivity, profile
    p = synth.make_small(nq=3)
    n = 12
    iq, w = np.arange(n, dtype=np.int32) % 3, np.linspace(0.2, 1.2, n)
    g = np.sqrt(np.where(np.arange(n) % 2, 20.0, 44.0)) * 2.0 * np.pi / p.cell.a
    ctx = context()
    try:
        states.load_problem(ctx, p)
        ctx.solve_batch(iq, w, g, p.eta, prec)
        info = ctx.batch_info()
        for _ in range(2):                               # the first profile also starts the profiler
            with profile(activities=[ProfilerActivity.CUDA, ProfilerActivity.CPU]) as prof:
                ctx.solve_batch(iq, w, g, p.eta, prec)
                torch.cuda.synchronize()
    finally:
        ctx.close()
    names = [e.name for e in prof.events() if e.device_type == torch.autograd.DeviceType.CUDA and "k_" in e.name]
    assert info["kernels_per_replay"] == len(names)
    assert info["solve_ctas"] == (n if prec == QCX_FP64 else 0)
    assert any("k_lu_head" in s for s in names) == (prec == QCX_FP64)
