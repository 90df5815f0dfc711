"""FP64 pair densities and overlaps of k points that differ by 1e-10 and 1e-12, as a list read from a file with ten decimals
beside a computed grid: the per-axis tables must keep such components apart (they merge only what differs by rounding).
The general kernels, which take every point's own components, are reached by adding irregular k points.

Tolerance: that of test_gpu_pair_tables (both sides evaluate the same closed form in FP64); a component moved by 1e-10
changes the phases of neighbouring cells by ~1e-9."""
import numpy as np
import pytest

import synth
from paper_2603_12326_gb300 import QCX_FP64
from tests.gpu_util import context, rel
from tests.test_gpu_pair_tables import A, LATTICES, _basis

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", ["fcc", "bcc"])
def test_close_points_keep_their_own_components(lattice):
    rng = np.random.default_rng(11)
    lat = LATTICES[lattice]
    reg = synth.kgrid(synth.Cell(lat, np.zeros((1, 3)), A), 4)
    reg = np.concatenate([reg, reg + [1e-10, -1e-10, 1e-10], reg + [1e-12, 1e-12, -1e-12]])
    k = np.concatenate([reg, rng.uniform(-0.5, 0.5, (1500, 3))])
    G = np.array([[0, 0, 0], [1, -2, 3]], np.int32)
    q = np.array([[0.11, 0.23, -0.31]])
    atoms, sa, sl, se = _basis("mixed")
    nb, nv, nc, n = int(np.sum(np.where(sl == 0, 1, 3))), 3, 5, len(k)
    Ck = synth.random_coeffs(rng, (n, nb, nv))
    Ckq = synth.random_coeffs(rng, (1, n, nb, nc))
    Ek, Ekq = rng.uniform(-1, 0, (n, nv)), rng.uniform(0.1, 1, (1, n, nc))
    out = {}
    ctx = context()
    try:
        ctx.set_basis(lat, atoms, sa, sl, se)
        for m in (len(reg), n):
            S = ctx.overlap(k[:m])[:len(reg)]
            ctx.set_states(k[:m], Ck[:m], Ek[:m], q, Ckq[:, :m], Ekq[:, :m])
            out[m] = S, ctx.pair_density(0, G, QCX_FP64, want=True)[:len(reg) * nv * nc]
    finally:
        ctx.close()
    for got, ref in zip(out[len(reg)], out[n]):
        assert rel(got, ref) < 1e-13
