"""The sizes at which the tests of a chi0 route compare results do take that route (the library chooses by estimated time,
so a changed estimate would leave such a test comparing another kernel)."""
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED, states
from tests import test_gpu_chi0_fp64_tc, test_gpu_chi0_panels, test_gpu_chi0_panels_cover, test_gpu_chi0_split
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


def _sizes(test):
    names, sizes = next(m for m in test.pytestmark if m.name == "parametrize").args
    return [dict(zip(names.split(","), s)) for s in sizes]


# narrow panels (0.13 eV, a few hundred of them); test_panels_match_fp64's own size at this eta is too small for the route
NARROW = dict(n_k=8, nv=4, nc=16, ng=181, nw=200, eta=0.1)
SMALL = dict(n_k=7, nv=3, nc=13, ng=181, nw=127, eta=0.1)
CASES = [("direct" if s == SMALL else "panels", QCX_MIXED, s)
         for s in _sizes(test_gpu_chi0_panels.test_panels_match_fp64) + [NARROW]] + \
        [("panels", QCX_MIXED, dict(s, eta=0.5)) for s in _sizes(test_gpu_chi0_panels_cover.test_cover_of_block_pairs)] + \
        [("fp64_slices", QCX_FP64, s) for s in _sizes(test_gpu_chi0_fp64_tc.test_sliced_chi0_matches_fp64)] + \
        [("direct", QCX_MIXED, s) for s in _sizes(test_gpu_chi0_split.test_split_chi0_matches_fp64)] + \
        [("fp64_sum", QCX_FP64, dict(n_k=2, nv=1, nc=3, ng=9, nw=4))]


@pytest.mark.parametrize("route,prec,size", CASES)
def test_sizes_take_their_route(route, prec, size):
    size = dict(size)
    eta = size.pop("eta", None)
    p = synth.make_tiny(nq=1, **size)
    if prec == QCX_MIXED:
        p.w = synth.omega_grid(40.0, size["nw"])
    if eta:
        p.eta = eta / synth.HARTREE_EV
    ctx = context()
    try:
        states.load_problem(ctx, p, [0])
        ctx.pair_density(0, p.G_int, prec)
        assert ctx.chi0_route(prec) is None
        ctx.chi0(0, p.w, p.eta, prec)
        assert ctx.chi0_route(prec) == route
        assert ctx.chi0_route(QCX_FP64 + QCX_MIXED - prec) is None
    finally:
        ctx.close()


def test_narrow_panels_match_fp64():
    test_gpu_chi0_panels.test_panels_match_fp64(**NARROW)
