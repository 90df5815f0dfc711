"""Device memory that a batch plan takes per distinct q: the rho planes (FP64: rho) and small arrays, not a set of pair-density
tables and work space (here ~55 MB in mixed precision) for each q.

The bound: the planes of one q and 8 MB for its small arrays (each allocation takes up to 2 MB)."""
import numpy as np
import pytest
import torch

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED, states
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [QCX_FP64, QCX_MIXED])
def test_memory_per_q(prec):
    p = synth.make_small()
    ctx = context()
    used, heads = {}, {}
    n = 20
    gmax = np.full(n, np.sqrt(48.0) * 2.0 * np.pi / p.cell.a)
    w = np.linspace(0.2, 1.2, n)
    try:
        states.load_problem(ctx, p)
        ctx.batch_autotune(False)
        for nq in (1, 2, 10):                            # the first call loads kernels
            iq = np.arange(n, dtype=np.int32) % nq
            ctx.solve_batch(iq[:1], w[:1], gmax[:1], p.eta, prec)   # a small plan in place of the last one
            free = torch.cuda.mem_get_info(0)[0]
            heads[nq] = ctx.solve_batch(iq, w, gmax, p.eta, prec)
            used[nq] = free - torch.cuda.mem_get_info(0)[0]
    finally:
        ctx.close()
    ng = int(max(heads[10][2]))
    planes = ng * p.nt * 16 if prec == QCX_FP64 else 3 * ((ng + 15) // 16 * 16) * 2 * p.nt * 2
    assert (used[10] - used[2]) / 8 < planes + (8 << 20)
    assert np.all(np.isfinite(heads[10][0]))


def test_inverse_in_groups_of_instances():
    """2600 instances of N_G = 335: their second copy for the inverse (0.9 MB each) is made for 1 GiB of them at a time.
    Per instance stay eps and the FP32 matrix, 24 N_G^2 bytes, the weights and vectors; the heads do not depend on the
    grouping beyond the launches' tiles."""
    p = synth.make_small(nq=1)
    ctx = context()
    used, heads = {}, {}
    g = np.sqrt(48.0) * 2.0 * np.pi / p.cell.a
    try:
        states.load_problem(ctx, p, [0])
        ctx.batch_autotune(False)
        for n in (100, 1300, 2600):
            w = np.linspace(0.2, 1.2, 2600)[:n]
            ctx.solve_batch(np.zeros(1, np.int32), w[:1], np.full(1, g), p.eta, QCX_MIXED)
            free = torch.cuda.mem_get_info(0)[0]
            heads[n] = ctx.solve_batch(np.zeros(n, np.int32), w, np.full(n, g), p.eta, QCX_MIXED)
            used[n] = free - torch.cuda.mem_get_info(0)[0]
    finally:
        ctx.close()
    ng = int(heads[100][2][0])
    assert (used[2600] - used[1300]) / 1300 < 24 * ng * (ng + 1) + 8 * p.nt + 256 * ng
    for n in (100, 1300):
        for i in range(2):
            assert np.max(np.abs(heads[2600][i][:n] / heads[n][i] - 1.0)) < 1e-6
