"""The blocked inverse at the edges of its panels (32 columns in FP32, 16 in FP64, narrower above N_G = 800) and
tiles (64), against numpy on the dielectric matrices formed from the exported chi0.

Tolerance: Gauss-Jordan with partial pivoting perturbs the inverse by a few n eps kappa_1 |A^-1| at most (the growth
factor of these matrices is O(1)); FP32 eps for the mixed path, where the matrix is rounded to FP32 first."""
import numpy as np
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED, states
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,unit", [(QCX_FP64, 2.0 ** -53), (QCX_MIXED, 2.0 ** -24)])
@pytest.mark.parametrize("ng", [1, 15, 16, 17, 32, 33, 64, 65, 127, 193, 330, 811])
def test_inverse_diagonal_at_panel_and_tile_edges(prec, unit, ng):
    p = synth.make_tiny(ng=ng, nw=3)
    ctx = context()
    try:
        states.load_problem(ctx, p, [0])
        ctx.pair_density(0, p.G_int, prec)
        chi = ctx.chi0(0, p.w, p.eta, prec, want=True)
        d, _, _ = ctx.invert_eps(0, prec)
    finally:
        ctx.close()
    vs = np.sqrt(4.0 * np.pi) / np.linalg.norm(p.qpts[0] + p.G_int @ p.cell.recip, axis=1)
    eps = np.eye(ng) - vs[:, None] * chi * vs
    inv = np.linalg.inv(eps)
    for a, x, got in zip(eps, inv, d):
        norm = np.abs(x).sum(axis=0).max()
        kappa = np.abs(a).sum(axis=0).max() * norm
        assert np.max(np.abs(got - np.diag(x))) <= 4.0 * ng * unit * kappa * norm + 1e-14
