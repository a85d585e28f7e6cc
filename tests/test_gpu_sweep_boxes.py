"""FP64 sweeps and factorisation with boxes of 4 layers, whose tiles of 3 layers hold lines
of two boxes, against the oracle's ILU(0) of the same boxes, through the C ABI.

Bars as in test_gpu_sweep_tiles.py: pivot inverses 1e-8 per entry of their family,
applies 1e-10 of the vector's largest entry; a line that takes a value across a cut, or
misses one within its box, gives errors of order one."""
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


# layers: one box; a box and one line; two boxes; three (the tiles' common edge); one line
# more; a ragged last box of each length
@pytest.mark.parametrize("nz", [4, 5, 8, 12, 13, 14, 15, 27])
@pytest.mark.parametrize("ny,ysub", [(9, 0), (19, 8)])
def test_apply_with_tiles_across_boxes(nz, ny, ysub):
    from paper_1910_06059_gb300 import Sim
    m = synth.small_model(5, ny, nz, wells=None)
    g, o = Sim(m), oracle.Oracle(m)
    g.subdomains, g.subdomains_z = ysub, 4
    o.set_subdomains(ysub, 4)
    st = synth.random_state(m, seed_member=5)
    for s in (g, o):
        s.set_state(*st)
        s.begin_step()
        s.assemble(2.0 * synth.DAY)
    dinv = g.factor()
    assert family_close(dinv, o.ilu0()[1], np.arange(o.n + 1), per_equation=False) <= 1e-8
    r = np.random.default_rng(12).normal(size=3 * g.n) * np.tile([1e-3, 1e-2, 1.0], g.n)
    z = g.precond_apply(r)
    assert vec_close(z, o.ilu_apply(r)) < 1e-10
    assert np.array_equal(g.precond_apply(r), z)
    g.close()


def test_boxes_of_four_layers_hold_no_more_than_one_box():
    """Tiles of 3 + 1 layers would take half as much again (28 MB here)."""
    from paper_1910_06059_gb300 import Sim
    held = []
    for sub in ((0, 0), (8, 4)):
        g = Sim(synth.small_model(40, 64, 48, wells=None))
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        if sub != (0, 0):
            g.subdomains_z = sub[1]
            g.subdomains = sub[0]
        torch.cuda.synchronize()
        held.append(before - torch.cuda.mem_get_info()[0])
        g.close()
    assert held[1] - held[0] <= 12 << 20
