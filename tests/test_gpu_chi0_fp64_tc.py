"""The FP64 chi0 on integer slices (tensor cores) at the edges of its tiles: N_G around 16, 64 and 128, frequency
groups of 8, K padding, and transitions in several chunks (the last case), against numpy's FP64 sum over the library's
own pair densities.

Tolerance: numpy's sum of N_t products carries at most N_t 2^-53 (about sqrt(N_t) 2^-53 in practice) of the sum of
magnitudes; the slices keep 61 bits below a row's maximum and no rounding in the sum.  1e-13 of the largest element
leaves a factor of a few over the former."""
import numpy as np
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64, states
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_k,nv,nc,ng,nw", [(6, 3, 7, 17, 40), (5, 2, 3, 16, 160), (5, 3, 5, 64, 9), (4, 2, 5, 65, 16),
                                             (3, 3, 3, 130, 9), (10, 5, 5, 531, 9)])
def test_sliced_chi0_matches_fp64(n_k, nv, nc, ng, nw):
    p = synth.make_tiny(n_k=n_k, nv=nv, nc=nc, ng=ng, nq=1, nw=nw)
    p.eta *= 0.1                                        # strong resonances: rows with a wide range of magnitudes
    ctx = context()
    try:
        states.load_problem(ctx, p, [0])
        rho = ctx.pair_density(0, p.G_int, QCX_FP64, want=True)
        chi = ctx.chi0(0, p.w, p.eta, QCX_FP64, want=True)
    finally:
        ctx.close()
    pick = np.unique(np.concatenate([np.arange(min(ng, 24)), np.arange(0, ng, 7), [ng - 1]]))
    r = rho[:, pick]
    dE = (p.Ekq[0][:, None, :] - p.Ek[:, :, None]).reshape(-1)
    for iw, w in enumerate(p.w):
        W = 1.0 / (w - dE + 1j * p.eta) - 1.0 / (w + dE + 1j * p.eta)
        ref = 2.0 / (p.nk * p.cell.volume) * ((r.conj().T * W) @ r)
        got = chi[iw][np.ix_(pick, pick)]
        assert np.max(np.abs(got - ref)) <= 1e-13 * np.max(np.abs(ref))
