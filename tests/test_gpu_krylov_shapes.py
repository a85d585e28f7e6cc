"""BiCGStab at the edges of its launches: less than a warp, one entry less and more than a block of
256 threads, both sides of the sizes above which the
blocks have 256 threads.

Bar: a solve that reports convergence at 1e-6 has ||R - J x|| <= 1e-6 ||R|| with the
residual formed here from the system that was read back, up to the rounding of the
products (n terms of 1e-16 |J| |x|, far below 1e-9 of ||R||)."""
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


# entries (3 a cell): 3, 255, 258, 765, 771; 65,520 and 65,550 (limit 65,536); cells: 256,
# 65,520 and 65,560 (limit 65,536)
@pytest.mark.parametrize("precond", ["ilu0", "cpr"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 17, 1), (43, 2, 1), (51, 5, 1), (257, 1, 1),
                                   (64, 4, 1), (56, 39, 10), (50, 23, 19), (56, 45, 26), (40, 149, 11)])
def test_solve_meets_its_tolerance(shape, precond):
    from paper_1910_06059_gb300 import Sim
    g = Sim(synth.small_model(*shape, wells=None))
    g.preconditioner = precond
    g.init_hydrostatic()
    g.begin_step()
    p, sw, x, flag, bhp = g.get_state()
    rng = np.random.default_rng(8)
    g.set_state(p * (1.0 + 1e-3 * rng.normal(size=g.n)), sw + 0.02 * rng.random(g.n), x, flag, bhp)
    g.assemble(2.0 * synth.DAY)
    g.factor()
    status, its, sol = g.solve(tol=1e-6, maxit=200)
    assert status == 0 and its >= 1
    rp, ci, J, R = g.system()
    row = np.repeat(np.arange(g.n), np.diff(rp))
    Jx = np.zeros((g.n, 3))
    np.add.at(Jx, row, np.einsum("eab,eb->ea", J, np.asarray(sol).reshape(g.n, 3)[ci]))
    assert np.linalg.norm(R - Jx) <= (1e-6 + 1e-9) * np.linalg.norm(R)
    g.close()
