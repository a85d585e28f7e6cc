"""The coarsest pressure solve of CPR's V-cycle (a cluster of 16 CTAs inverts the
operator, columns dealt out in turn) at the sizes where the dealing has edges,
through the C ABI.

A model of at most 200 cells has a single level, so its V-cycle is the coarsest
solve alone: x = A_p^-1 b.  Bar: the residual b - A_p x against |A_p| |x| + |b|,
entry by entry, n x 1e-13 (backward error of Gauss-Jordan with partial pivoting
on these row-dominant matrices, a few units of rounding per elimination step)."""
from __future__ import annotations

import numpy as np
import pytest

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


def _dense(ap, nx, ny, nz):
    n = nx * ny * nz
    A = np.zeros((n, n))
    c = np.arange(n)
    i, j, k = c % nx, c // nx % ny, c // (nx * ny)
    has = [i >= 0, i > 0, i + 1 < nx, j > 0, j + 1 < ny, k > 0, k + 1 < nz]
    for b, d in enumerate((0, -1, 1, -nx, nx, -nx * ny, nx * ny)):
        A[c[has[b]], c[has[b]] + d] = ap[has[b], b]
    return A


# one column per CTA or none (1, 3, 15), exactly one (16), one more (17), two
# (32), a row more than a CTA's threads never occurs below 200; the largest (200)
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 1, 1), (5, 3, 1), (4, 4, 1), (17, 1, 1),
                                   (4, 4, 2), (11, 3, 3), (10, 10, 2), (199, 1, 1)])
def test_single_level_vcycle_is_the_exact_solve(shape):
    from paper_1910_06059_gb300 import Sim
    m = synth.small_model(*shape, wells=None)
    g = Sim(m)
    g.preconditioner = "cpr"
    g.set_state(*synth.random_state(m, seed_member=2))
    g.begin_step()
    g.assemble(2.0 * synth.DAY)
    g.factor()
    sizes, _ = g.cpr_hierarchy()
    assert sizes == [g.n]
    _, ap = g.cpr_pressure_system()
    A = _dense(ap, *shape)
    b = np.random.default_rng(4).normal(size=g.n)
    x = g.cpr_vcycle(b)
    res = np.abs(b - A @ x)
    assert np.all(res <= g.n * 1e-13 * (np.abs(A) @ np.abs(x) + np.abs(b)))
    g.close()
