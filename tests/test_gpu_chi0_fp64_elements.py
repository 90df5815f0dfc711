"""Every element of the FP64 chi0 against sums in extended precision over the library's own pair densities, with resonances
from wide to far narrower than any physical one: the slices hold a row's values to 2^-61 of its largest, up to 1/eta.

Tolerance per element, over sum |rho||W||rho|: N_t 2^-53 for the sum of N_t rounded products in any order, and 8 2^-53 for
the rounding of W and of the products themselves."""
import numpy as np
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64, states
from tests.gpu_util import context

pytestmark = pytest.mark.gpu
L = np.longdouble


@pytest.mark.parametrize("eta", [4e-3, 4e-5, 1e-7, 1e-12])
def test_every_element(eta):
    p = synth.make_tiny(n_k=4, nv=3, nc=5, ng=33, nq=1, nw=6)
    dE = (p.Ekq[0][:, None, :] - p.Ek[:, :, None]).reshape(-1)
    w = p.w.copy()
    w[2], w[4] = dE[320], dE[500] + eta                  # on a resonance and on its flank
    ctx = context()
    try:
        states.load_problem(ctx, p, [0])
        rho = ctx.pair_density(0, p.G_int, QCX_FP64, want=True)
        chi = ctx.chi0(0, w, eta, QCX_FP64, want=True)
        assert ctx.chi0_route(QCX_FP64) == "fp64_slices"
    finally:
        ctx.close()
    r, i, pref = rho.real.astype(L), rho.imag.astype(L), L(2.0 / (p.nk * p.cell.volume))
    e = L(eta)
    for n in range(len(w)):
        a, b = L(w[n]) - dE.astype(L), L(w[n]) + dE.astype(L)
        x, y = a / (a * a + e * e) - b / (b * b + e * e), e / (b * b + e * e) - e / (a * a + e * e)
        xr, xi = x[:, None] * r - y[:, None] * i, x[:, None] * i + y[:, None] * r
        re, im = pref * (r.T @ xr + i.T @ xi), pref * (r.T @ xi - i.T @ xr)
        err = np.hypot((chi[n].real.astype(L) - re).astype(float), (chi[n].imag.astype(L) - im).astype(float))
        size = float(pref) * ((np.abs(rho).T * np.hypot(x, y).astype(float)) @ np.abs(rho))
        assert np.all(err <= (p.nt + 8) * 2.0 ** -53 * size)
