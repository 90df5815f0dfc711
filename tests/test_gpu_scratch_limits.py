"""Routes that have another to fall back on (chi0 through energy panels and integer slices, pair-density tables) where device
memory is short: what a call cannot do without is allocated first or gets their buffers back, a route that does not fit
keeps nothing, and the results are those of an unlimited run (of the other route: its documented error).

The memory is taken by one large allocation that leaves a chosen amount; the amounts follow from the sizes of the buffers
(eps N_w N_G^2 16 bytes, weights, FP64 sums of the direct kernel, inverse), 16 MB allowed for small ones."""
import numpy as np
import pytest
import torch

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED, states
from tests.gpu_util import context, rel, rel_spectrum

pytestmark = pytest.mark.gpu
MB = 1 << 20


def _free():
    return torch.cuda.mem_get_info(0)[0]


class _Leave:
    """Takes all device memory but `bytes` while the block runs."""

    def __init__(self, n):
        self.n = n

    def __enter__(self):
        torch.cuda.empty_cache()
        self.t = torch.empty(_free() - self.n, dtype=torch.uint8, device="cuda")

    def __exit__(self, *exc):
        del self.t
        torch.cuda.empty_cache()


@pytest.fixture(scope="module")
def kernels():
    """Kernels load at their first launch and need memory then: one small pass by every route."""
    for size in (dict(n_k=2, nv=1, nc=3, ng=9, nw=4), dict(n_k=3, nv=2, nc=3, ng=33, nw=9)):
        p = synth.make_tiny(nq=1, **size)
        ctx = context()
        states.load_problem(ctx, p, [0])
        for prec in (QCX_FP64, QCX_MIXED):
            ctx.pair_density(0, p.G_int, prec)
            ctx.chi0(0, p.w, p.eta, prec)
            ctx.invert_eps(0, prec)
        ctx.close()


def _problem(n_k, nc, nw):
    p = synth.make_tiny(n_k=n_k, nv=4, nc=nc, ng=181, nq=1, nw=nw)
    p.w = synth.omega_grid(40.0, nw)
    return p


def _direct(p, nw):
    """eps; weights and FP64 sums of the direct kernel; both with the inverse and its smallest second copy."""
    eps = nw * 181 * 181 * 16
    chi = nw * p.nt * 8 + 3 * nw * 128 * 192 * 8
    return eps, eps + chi, eps + chi + eps // 2


def test_panels_that_do_not_fit_leave_nothing_behind(kernels):
    p = _problem(8, 16, 200)
    loss = []
    for limited in (False, True):
        ctx = context()
        try:
            states.load_problem(ctx, p, [0])
            ctx.pair_density(0, p.G_int, QCX_MIXED)
            _, chi, all_ = _direct(p, 200)
            with _Leave(all_ + 40 * MB if limited else _free() - 2 * MB):
                free = _free()
                ctx.chi0(0, p.w, p.eta, QCX_MIXED)
                if limited:
                    assert free - _free() < chi + 16 * MB
                ctx.invert_eps(0, QCX_MIXED, want=False)
                loss.append(ctx.loss_function(0, QCX_MIXED))
        finally:
            ctx.close()
    for a, b in zip(loss[1], loss[0]):
        assert rel_spectrum(a, b) < 1e-4


def test_slices_that_do_not_fit_leave_nothing_behind(kernels):
    p = _problem(6, 12, 8)
    chi0 = []
    for limited in (False, True):
        ctx = context()
        try:
            states.load_problem(ctx, p, [0])
            ctx.pair_density(0, p.G_int, QCX_FP64)
            with _Leave(400 * MB if limited else _free() - 2 * MB):
                free = _free()
                ctx.chi0(0, p.w, p.eta, QCX_FP64)
                if limited:
                    assert free - _free() < _direct(p, 8)[0] + 16 * MB
            chi0.append(ctx.chi0(0, p.w, p.eta, QCX_FP64, want=True))
        finally:
            ctx.close()
    assert rel(chi0[1], chi0[0]) < 1e-12


def test_tables_come_after_rho(kernels):
    p = _problem(8, 16, 8)
    rho = []
    for limited in (False, True):
        ctx = context()
        try:
            states.load_problem(ctx, p, [0])
            planes = 3 * 192 * 2 * p.nt * 2
            with _Leave(planes + 24 * MB if limited else _free() - 2 * MB):
                ctx.pair_density(0, p.G_int, QCX_MIXED)
            rho.append(ctx.pair_density(0, p.G_int, QCX_MIXED, want=True))
        finally:
            ctx.close()
    assert rel(rho[1], rho[0]) < 1e-5


def test_dead_buffers_are_given_back(kernels):
    p = _problem(8, 16, 200)
    loss = []
    for limited in (False, True):
        ctx = context()
        try:
            states.load_problem(ctx, p, [0])
            ctx.pair_density(0, p.G_int, QCX_MIXED)
            ctx.chi0(0, p.w, p.eta, QCX_MIXED)           # the panels' buffers hold several times the inverse's
            with _Leave(16 * MB if limited else _free() - 2 * MB):
                ctx.invert_eps(0, QCX_MIXED, want=False)
                loss.append(ctx.loss_function(0, QCX_MIXED))
        finally:
            ctx.close()
    for a, b in zip(loss[1], loss[0]):
        assert rel_spectrum(a, b) < 1e-6
