"""Pair densities and overlaps from the per-axis tables against the kernels that form every lattice sum, over the forms
the tables accept: lattices with one, two and four characters, s-only, p-only and mixed shells, band counts around the
register blocks, odd sizes.  The general kernels are reached by adding irregular k points, for which tables would not
save work; the regular points come first in both calls.

Tolerance: both sides evaluate the same closed form; FP64 to a few hundred roundings of the largest element, FP32 to
1e-5 of it (the sums over ~N_b^2 terms of either side carry ~1e-6)."""
import numpy as np
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64, QCX_MIXED
from tests.gpu_util import context, rel

pytestmark = pytest.mark.gpu

A = 10.0
LATTICES = {"sc": A * np.eye(3), "fcc": 0.5 * A * np.array([[0.0, 1, 1], [1, 0, 1], [1, 1, 0]]),
            "bcc": 0.5 * A * np.array([[-1.0, 1, 1], [1, -1, 1], [1, 1, -1]])}


def _basis(kind):
    atoms = np.array([[0.0, 0.0, 0.0], [2.3, 2.1, 2.7]])
    shells = {"s": [(0, 0, 0.4), (1, 0, 0.9)], "p": [(0, 1, 0.5), (1, 1, 1.1)],
              "mixed": [(0, 0, 0.4), (0, 1, 0.4), (0, 0, 3.0), (1, 1, 0.8), (1, 0, 40.0), (1, 1, 40.0)]}[kind]
    a, l, e = zip(*shells)
    return atoms, np.array(a, np.int32), np.array(l, np.int32), np.array(e)


@pytest.mark.parametrize("lattice,shells,nv,nc", [("fcc", "mixed", 4, 5), ("fcc", "s", 1, 1), ("fcc", "p", 3, 7),
                                                  ("sc", "mixed", 5, 9), ("bcc", "mixed", 9, 33), ("bcc", "p", 16, 3)])
def test_tables_match_general_kernels(lattice, shells, nv, nc):
    rng = np.random.default_rng(5)
    lat = LATTICES[lattice]
    cell = synth.Cell(lat, np.zeros((1, 3)), A)
    reg = synth.kgrid(cell, 4)
    extra = rng.uniform(-0.5, 0.5, (500, 3))
    G = np.array([[0, 0, 0], [1, -2, 3]], np.int32)      # two values per axis: irregular k points then reject the tables
    q = np.array([[0.11, 0.23, -0.31]])
    atoms, sa, sl, se = _basis(shells)
    nb = int(np.sum(np.where(sl == 0, 1, 3)))
    n = len(reg) + len(extra)
    Ck = synth.random_coeffs(rng, (n, nb, nv))
    Ckq = synth.random_coeffs(rng, (1, n, nb, nc))
    Ek, Ekq = rng.uniform(-1, 0, (n, nv)), rng.uniform(0.1, 1, (1, n, nc))
    out = {}
    ctx = context()
    try:
        ctx.set_basis(lat, atoms, sa, sl, se)
        for name, m in (("tab", len(reg)), ("gen", n)):
            k = np.concatenate([reg, extra])[:m]
            out[name, "S"] = ctx.overlap(k)[:len(reg)]
            ctx.set_states(k, Ck[:m], Ek[:m], q, Ckq[:, :m], Ekq[:, :m])
            for prec in (QCX_FP64, QCX_MIXED):
                out[name, prec] = ctx.pair_density(0, G, prec, want=True)[:len(reg) * nv * nc]
    finally:
        ctx.close()
    assert rel(out["tab", "S"], out["gen", "S"]) < 1e-13
    assert rel(out["tab", QCX_FP64], out["gen", QCX_FP64]) < 1e-13
    assert rel(out["tab", QCX_MIXED], out["gen", QCX_FP64]) < 1e-5
