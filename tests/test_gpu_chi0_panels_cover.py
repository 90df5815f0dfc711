"""The energy panels' cover of the pairs of 64-row G' blocks (tiles whose columns wrap around the last block, S below the
diagonal written as its conjugate) at block counts 3, 4 and 7 with last blocks of 16 to 64 rows, against the FP64 path,
with the tolerance of test_gpu_chi0_panels; and the barrier protocol of the longer ring on the CPU."""
import numpy as np
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED, states
from tests.gpu_util import context, rel
from tests.test_chi0_panels_protocol import _constant
from tests.test_chi0_protocol import _run


@pytest.mark.gpu
@pytest.mark.parametrize("n_k,nv,nc,ng,nw", [(6, 4, 12, 129, 120), (6, 3, 11, 176, 128), (6, 4, 9, 192, 120),
                                             (6, 3, 10, 256, 80), (6, 2, 9, 395, 100)])
def test_cover_of_block_pairs(n_k, nv, nc, ng, nw):
    p = synth.make_tiny(n_k=n_k, nv=nv, nc=nc, ng=ng, nq=1, nw=nw)
    p.eta = 0.5 / synth.HARTREE_EV
    p.w = synth.omega_grid(40.0, nw)
    chi = {}
    ctx = context()
    try:
        states.load_problem(ctx, p, [0])
        for prec in (QCX_FP64, QCX_MIXED):
            ctx.pair_density(0, p.G_int, prec)
            chi[prec] = ctx.chi0(0, p.w, p.eta, prec, want=True)
    finally:
        ctx.close()
    for iw in range(0, nw, 9):
        a, b = chi[QCX_MIXED][iw], chi[QCX_FP64][iw]
        assert rel(a, b) < 3e-6
        # every 64-block pair on its own: a block left out or written twice is wrong by its own size
        for i in range(0, ng, 64):
            for j in range(0, ng, 64):
                assert np.max(np.abs((a - b)[i:i + 64, j:j + 64])) < 3e-6 * np.max(np.abs(b))


@pytest.mark.parametrize("kstages", [1, 2, 5, 8])
@pytest.mark.parametrize("fault", [{}, {"timeouts": True}, {"withhold": True, "timeouts": True}])
def test_protocol_of_the_longer_ring(kstages, fault):
    for seed in range(6):
        errors, aborted = _run(kstages, _constant("PG_NSTAGE") + 1, _constant("PG_PROMOTE"), seed, ngroups=1, ntile=6,
                               drain_warps=8, **fault)
        assert not errors, (kstages, seed, errors[:3])
        assert bool(aborted) <= bool(fault)
