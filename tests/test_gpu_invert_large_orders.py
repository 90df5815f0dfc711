"""The blocked inverse where a thread of the panel holds more than one row (orders above 1024, up to the 4096 that the library
takes, panels down to two columns) and where the matrices need more than one group (a second copy above 1 GiB).

Against numpy with the tolerance of test_gpu_invert_blocked."""
import numpy as np
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED, states
from tests.gpu_util import context

pytestmark = pytest.mark.gpu
UNIT = {QCX_FP64: 2.0 ** -53, QCX_MIXED: 2.0 ** -24}


def _check(prec, ng, nw, pick):
    p = synth.make_tiny(ng=ng, nw=nw)
    ctx = context()
    try:
        states.load_problem(ctx, p, [0])
        ctx.pair_density(0, p.G_int, prec)
        chi = ctx.chi0(0, p.w, p.eta, prec, want=True)
        d, _, _ = ctx.invert_eps(0, prec)
    finally:
        ctx.close()
    vs = np.sqrt(4.0 * np.pi) / np.linalg.norm(p.qpts[0] + p.G_int @ p.cell.recip, axis=1)
    for w in pick:
        a = np.eye(ng) - vs[:, None] * chi[w] * vs
        x = np.linalg.inv(a)
        norm = np.abs(x).sum(axis=0).max()
        kappa = np.abs(a).sum(axis=0).max() * norm
        assert np.max(np.abs(d[w] - np.diag(x))) <= 4.0 * ng * UNIT[prec] * kappa * norm + 1e-14


@pytest.mark.parametrize("prec", [QCX_FP64, QCX_MIXED])
@pytest.mark.parametrize("ng", [1025, 2081, 4096])
def test_orders_with_several_rows_per_thread(prec, ng):
    _check(prec, ng, 1, [0])


@pytest.mark.parametrize("prec,ng,nw", [(QCX_FP64, 1100, 60), (QCX_MIXED, 1100, 115)])
def test_groups_of_matrices(prec, ng, nw):
    per = (1 << 30) // (ng * ng * (16 if prec == QCX_FP64 else 8))
    assert 1 < per < nw - 1
    _check(prec, ng, nw, [0, per - 1, per, nw - 1])
