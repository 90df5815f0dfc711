"""Contexts of different sizes used by several host threads at once: every call succeeds and gives the bits of the same call
made alone."""
import threading

import numpy as np
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED, states
from tests.gpu_util import context

pytestmark = pytest.mark.gpu
SIZES = [dict(n_k=2, nv=2, nc=3, ng=9, nw=4, shells_per_atom=2), dict(n_k=2, nv=4, nc=6, ng=65, nw=6, shells_per_atom=5),
         dict(n_k=2, nv=3, nc=5, ng=33, nw=3, shells_per_atom=3)]


def _pass(ctx, p):
    out = [ctx.overlap(p.kpts)]
    for prec in (QCX_FP64, QCX_MIXED):
        ctx.pair_density(0, p.G_int, prec)
        out += [ctx.chi0(0, p.w, p.eta, prec, want=True), ctx.invert_eps(0, prec)[0], *ctx.loss_function(0, prec)]
    return out


def test_contexts_in_threads():
    work, errors = [], []
    for size in SIZES:
        p = synth.make_tiny(nq=1, **size)
        ctx = context()
        states.load_problem(ctx, p, [0])
        work.append((ctx, p, _pass(ctx, p)))

    def run(ctx, p, want):
        try:
            for _ in range(1500):
                for a, b in zip(_pass(ctx, p), want):
                    assert np.array_equal(a, b)
        except Exception as e:                           # noqa: BLE001 - reported below
            errors.append(e)

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for ctx, *_ in work:
        ctx.close()
    assert not errors, errors
