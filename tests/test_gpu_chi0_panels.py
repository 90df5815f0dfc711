"""The mixed chi0 through energy panels (many frequencies) against the FP64 path on the same states, at the edges of its
tiling: N_G around 32, 64 and 192 (column chunks with and without their own rows), panels of a few and of more than
2048 transitions (segments), ragged transitions and frequencies.

Tolerance: the mixed path's documented error of chi0 (1e-6 of the largest element, from the FP32 pair densities and the
FP32 windows; 3e-6 allowed) and its 1e-4 bar on the loss where it exceeds 1e-3 of a spectrum's maximum."""
import numpy as np
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED, states
from tests.gpu_util import context, rel, rel_spectrum

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_k,nv,nc,ng,nw,eta", [(6, 4, 12, 65, 200, 0.5), (6, 3, 11, 193, 65, 0.5), (8, 4, 16, 33, 200, 3.0),
                                                 (7, 3, 13, 181, 127, 0.1), (6, 5, 9, 290, 64, 1.0), (5, 7, 15, 17, 900, 0.2)])
def test_panels_match_fp64(n_k, nv, nc, ng, nw, eta):
    p = synth.make_tiny(n_k=n_k, nv=nv, nc=nc, ng=ng, nq=1, nw=nw)
    p.eta = eta / synth.HARTREE_EV
    p.w = synth.omega_grid(40.0, nw)                     # inside the transitions: no isolated poles above them
    out = {}
    ctx = context()
    try:
        states.load_problem(ctx, p, [0])
        for prec in (QCX_FP64, QCX_MIXED):
            ctx.pair_density(0, p.G_int, prec)
            chi = ctx.chi0(0, p.w, p.eta, prec, want=True)
            d, e, _ = ctx.invert_eps(0, prec)
            out[prec] = (chi, d, e, *ctx.loss_function(0, prec))
    finally:
        ctx.close()
    for iw in range(0, nw, max(1, nw // 40)):
        assert rel(out[QCX_MIXED][0][iw], out[QCX_FP64][0][iw]) < 3e-6
    assert rel_spectrum(out[QCX_MIXED][3], out[QCX_FP64][3]) < 1e-4
    assert rel_spectrum(out[QCX_MIXED][4], out[QCX_FP64][4]) < 1e-4
