"""Factorisation and FP64 triangular sweeps at the edges of their tiles (4 x 3 x-lines, levels in
rings of 8, a ticket per tile) against the oracle's ILU(0), through the C ABI.

Bars: pivot inverses 1e-8 per entry of their family (the conditioning argument of
test_gpu_subdomains.py); applies 1e-10 of the vector's largest entry, as for the other applies on random
states (two FP64 factorisations that sum in different orders differ by about
cond(D) x 1.1e-16); a neighbour value that is missing, stale or taken from the
wrong line gives errors of order one.  A repeated apply gives the same bits."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from helpers import family_close, vec_close

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1910_06059_gb300.build import build
    build()


# grid, block-Jacobi boxes
SHAPES = [
    ((1, 1, 1), (0, 0)),        # one cell: 6 levels, fewer than a ring
    ((1, 4, 3), (0, 0)),        # one full tile, one cell deep
    ((2, 5, 4), (0, 0)),        # one line past a tile in j and k
    ((9, 3, 2), (0, 0)),        # one ragged tile, levels past one ring
    ((11, 8, 6), (0, 0)),       # full tiles, 16 levels: two rings exactly
    ((12, 9, 7), (0, 0)),       # one level past two rings, ragged in j and k
    ((3, 125, 31), (0, 0)),     # 352 tiles, more than two CTAs on each of 152 SMs
    ((7, 22, 11), (8, 4)),      # boxes of 4 layers (tiles of 3 and 1), a ragged last box
    ((5, 17, 23), (16, 8)),     # boxes of 8 layers (3, 3, 2), a one-line last slab
    ((6, 21, 9), (0, 4)),       # cuts in z only
]


@pytest.mark.parametrize("shape,sub", SHAPES)
def test_apply_at_tile_edges(shape, sub):
    from paper_1910_06059_gb300 import Sim
    m = synth.small_model(*shape, wells=None)
    g, o = Sim(m), oracle.Oracle(m)
    if sub != (0, 0):
        g.subdomains = sub[0]
        g.subdomains_z = sub[1]
        o.set_subdomains(*sub)
    st = synth.random_state(m, seed_member=3)
    for s in (g, o):
        s.set_state(*st)
        s.begin_step()
        s.assemble(2.0 * synth.DAY)
    dinv = g.factor()
    assert family_close(dinv, o.ilu0()[1], np.arange(o.n + 1), per_equation=False) <= 1e-8
    r = np.random.default_rng(11).normal(size=3 * g.n) * np.tile([1e-3, 1e-2, 1.0], g.n)
    z = g.precond_apply(r)
    assert vec_close(z, o.ilu_apply(r)) < 1e-10
    for _ in range(3):
        assert np.array_equal(g.precond_apply(r), z)
    g.close()
