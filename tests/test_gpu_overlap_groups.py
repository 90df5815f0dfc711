"""The overlap from the tables walks the pairs of shell groups as rows r and n - 1 - r of a triangle: 1 to 5 groups (odd
numbers have a middle row) against the kernel that forms every lattice sum, which an irregular k list takes; tolerance of
test_gpu_pair_tables."""
import numpy as np
import pytest

import synth
from tests.gpu_util import context, rel
from tests.test_gpu_pair_tables import A, LATTICES

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ngrp", [1, 2, 3, 4, 5])
def test_overlap_of_any_number_of_groups(ngrp):
    lat = LATTICES["fcc"]
    atoms = np.array([[0.0, 0.0, 0.0], [2.3, 2.1, 2.7]])
    sa = np.repeat(np.arange(ngrp) % 2, 2).astype(np.int32)
    order = np.argsort(sa, kind="stable")
    sl, se = np.tile([0, 1], ngrp).astype(np.int32), np.repeat(0.4 * 1.7 ** np.arange(ngrp), 2)
    reg = synth.kgrid(synth.Cell(lat, np.zeros((1, 3)), A), 4)
    extra = np.random.default_rng(3).uniform(-0.5, 0.5, (1500, 3))
    ctx = context()
    try:
        ctx.set_basis(lat, atoms, sa[order], sl[order], se[order])
        tab = ctx.overlap(reg)
        gen = ctx.overlap(np.concatenate([reg, extra]))[:len(reg)]
    finally:
        ctx.close()
    assert rel(tab, gen) < 1e-13
