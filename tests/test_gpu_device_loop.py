"""BiCGStab's device-side loop against the graph that the host replays (used while timing
is on): the same kernels on the same numbers, so the same bits, iterations, restarts and
status at the iteration limit, at convergence in either half step, over restarts and with
nothing to solve."""
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


def _both(g, **kw):
    out = []
    for timed in (False, True):
        g.set_timing(timed)
        st, its, x, info = g.solve(report=True, **kw)
        out.append((st, its, info, x.copy()))
    g.set_timing(False)
    (s0, i0, r0, x0), (s1, i1, r1, x1) = out
    assert (s0, i0, r0) == (s1, i1, r1)
    assert np.array_equal(x0, x1)
    return s0, i0, r0


@pytest.mark.parametrize("precond", ["ilu0", "cpr"])
@pytest.mark.parametrize("wells", ["reduced", "standard"])
def test_loop_equals_the_replayed_graph(precond, wells):
    from paper_1910_06059_gb300 import Sim
    m = synth.small_model(21, 18, 11, wells="5spot")
    g = Sim(m)
    g.set_well_model(wells)
    g.preconditioner = precond
    g.init_hydrostatic()
    g.begin_step()
    p, sw, x, flag, bhp = g.get_state()
    rng = np.random.default_rng(8)
    g.set_state(p * (1.0 + 1e-3 * rng.normal(size=g.n)), sw + 0.02 * rng.random(g.n), x, flag, bhp)
    g.assemble(2.0 * synth.DAY)
    g.factor()
    for maxit in (1, 2, 3, 4, 5, 8, 9):              # the replayed graph has four iterations
        st, its, info = _both(g, tol=1e-15, maxit=maxit)
        assert its <= maxit
        if its == maxit:
            assert st != 0
    ended = set()
    for tol in (0.5, 0.1, 1e-2, 1e-3, 1e-5, 1e-8):
        st, its, info = _both(g, tol=tol, maxit=400)
        assert st == 0 and its >= 1 and info["rel_res"] <= tol
        ended.add(its)
    assert len(ended) >= 3
    # below what one recurrence reaches: restarts from the true residual, then giving up
    st, its, info = _both(g, tol=1e-17, maxit=400)
    assert st != 0 and info["restarts"] >= 1
    st, its, info = _both(g, tol=1e-3, maxit=400)    # and the next solve starts anew
    assert st == 0 and info["restarts"] == 0
    g.close()
