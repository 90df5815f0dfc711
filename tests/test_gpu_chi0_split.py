"""The direct mixed chi0 with K splits (fewer CTAs than SMs, or a little over a wave) against the FP64 path: one to a few
hundred CTAs, ragged last splits, N_G with one and two column chunks.  Tolerance: as for the kernel without splits (3e-6 of
the largest element; the splits add FP64 sums)."""
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED, states
from tests.gpu_util import context, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_k,nv,nc,ng,nw", [(4, 3, 5, 13, 1), (4, 4, 12, 27, 50), (3, 5, 13, 113, 37), (3, 3, 11, 64, 160),
                                             (4, 2, 7, 65, 90), (3, 4, 9, 201, 5)])
def test_split_chi0_matches_fp64(n_k, nv, nc, ng, nw):
    p = synth.make_tiny(n_k=n_k, nv=nv, nc=nc, ng=ng, nq=1, nw=nw)
    out = {}
    ctx = context()
    try:
        states.load_problem(ctx, p, [0])
        for prec in (QCX_FP64, QCX_MIXED):
            ctx.pair_density(0, p.G_int, prec)
            out[prec] = ctx.chi0(0, p.w, p.eta, prec, want=True), ctx.invert_eps(0, prec)[1]
    finally:
        ctx.close()
    for iw in range(nw):
        assert rel(out[QCX_MIXED][0][iw], out[QCX_FP64][0][iw]) < 3e-6
    assert rel(out[QCX_MIXED][1], out[QCX_FP64][1]) < 3e-6
