"""Assembly and convergence measures at the edges of their blocks (64 cells a block, a thread
per face, a warp per well and 32 connections, up to 1024 blocks of partial sums) against the oracle.

Bar: 1e-12 K for the residual, K_a = sum_s |J_as| |y_s| over the cell's diagonal
block.  K bounds the terms that cancel in a residual (a face's mobility times the
pressures, the accumulated volumes up to 1 / s_w <= 9), and some 200 roundings of
1.1e-16 in the cell's functions come to 2e-13 of them.  A face or connection that
is missing, doubled or of the wrong sign is of order K.  The blocks by the same
bar after multiplying with y; the measures by the bar of the sums and maxima they
are taken from."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1910_06059_gb300.build import build
    build()
    oracle.build()


# axes of one cell, blocks of 63, 64 and 65 cells, wells with 7, 33 and 70
# connections, and more than 1024 blocks (70,200 cells)
@pytest.mark.parametrize("shape,wells", [
    ((1, 1, 1), None), ((64, 1, 1), None), ((1, 65, 1), None), ((1, 5, 7), "5spot"),
    ((7, 1, 9), "5spot"), ((4, 4, 4), "gas"), ((5, 4, 33), "5spot"), ((3, 4, 70), "5spot"),
    ((60, 45, 26), "5spot")])
def test_assembly_and_norms_match_oracle(shape, wells):
    from paper_1910_06059_gb300 import Sim
    m = synth.small_model(*shape, wells=wells)
    dt = 2.0 * synth.DAY
    g, o = Sim(m), oracle.Oracle(m)
    for s in (g, o):
        s.set_state(*synth.random_state(m, seed_member=5))
        s.begin_step()
        s.set_state(*synth.random_state(m, seed_member=6))
        s.assemble(dt)
    rp, ci, J, R = g.system()
    rpo, cio, Jo, Ro = o.system()
    assert np.array_equal(rp, rpo) and np.array_equal(ci, cio)
    row = np.repeat(np.arange(g.n), np.diff(rp))
    p, sw, x, _, _ = o.get_state()[:5]
    y = np.stack([p, sw, np.maximum(np.abs(x), 1e-2)], axis=1)
    D = Jo[ci == row]
    assert len(D) == g.n
    K = np.einsum("cas,cs->ca", np.abs(D), y)
    assert np.all(np.abs(R - Ro) <= 1e-12 * K)
    assert np.all(np.abs(J - Jo) * y[ci][:, None, :] <= 1e-12 * (K[row] + K[ci])[:, :, None])
    N, No = g.norms(dt), o.norms(dt)
    pv = g.get_static()["pv"]
    worst = (np.abs(Ro) / pv[:, None]).max(axis=0)
    scale = No[3:6] / worst                    # dt times the mean of 1 / b
    assert np.all(np.abs(N[:3] - No[:3]) <= 1e-12 * scale * K.sum(axis=0) / pv.sum())
    assert np.all(np.abs(N[3:6] - No[3:6]) <= 1e-12 * scale * (K / pv[:, None]).max(axis=0))
    if wells is not None:
        target = abs(m["wells"][0]["target"])
        assert abs(N[6] - No[6]) <= 1e-12 * K.sum() / target
    g.close()
