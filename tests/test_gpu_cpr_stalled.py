"""CPR's V-cycle when aggregation stalls above its usual coarsest size: cells that
nothing connects stay alone on every level.  The coarsest operator then has more rows
than the cluster inverse has threads (256), or is too large for it (512) and goes to the
one-CTA form.

The reference is the oracle's V-cycle on the operator and the hierarchy that the
simulator reports.  Bar: 1e-10 of the vector's largest entry, as for the other V-cycles,
and n eps cond(A_c) for the dense inverse (both sides eliminate in their own order).  A
transposed inverse misses it by far, which is checked on the oracle."""
from __future__ import annotations

import numpy as np
import pytest
import scipy.sparse as sp

import synth
from helpers import make_model
from oracle.cpr import AMG

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1910_06059_gb300.build import build
    build()


def _vcycle_error(amg, coarse, b, x):
    keep, amg.coarse = amg.coarse, coarse
    y = amg.vcycle(b)
    amg.coarse = keep
    return float(np.max(np.abs(x - y)) / np.max(np.abs(y)))


# a chain that leaves about ten unknowns after eleven aggregations, and cells on their own
@pytest.mark.parametrize("alone,large", [(300, False), (490, False), (560, True)])
def test_vcycle_on_a_stalled_hierarchy(alone, large):
    from paper_1910_06059_gb300 import Sim
    n = 200_000
    rng = np.random.default_rng(9)
    perm = 1e-13 * np.exp(2.0 * rng.normal(size=n))
    perm[:alone] = 1e-200                     # T = k^2 / 2k underflows to zero between these
    m = make_model(n, 1, 1, perm, 0.2, [])
    g = Sim(m)
    g.preconditioner = "cpr"
    g.init_hydrostatic()
    g.begin_step()
    g.assemble(1e4 * synth.DAY)               # the aggregates are coupled on the last level
    g.factor()
    sizes, maps = g.cpr_hierarchy()
    assert len(sizes) == 12 and alone <= sizes[-1] <= alone + 40
    assert (sizes[-1] > 512) == large and sizes[-1] > 256
    _, ap = g.cpr_pressure_system()
    A = sp.diags([ap[:, 0], ap[1:, 1], ap[:-1, 2]], [0, -1, 1], format="csr")
    Ps = [sp.csr_matrix((np.ones(len(a)), (np.arange(len(a)), a)), shape=(len(a), nc))
          for a, nc in zip(maps, sizes[1:])]
    amg = AMG(A, prolongators=Ps)
    b = rng.normal(size=n)
    x = g.cpr_vcycle(b)
    bar = 1e-10 + sizes[-1] * 2.0 ** -52 * np.linalg.cond(amg.A[-1].toarray())
    assert _vcycle_error(amg, amg.coarse.T, b, x) > 100 * bar
    assert _vcycle_error(amg, amg.coarse, b, x) <= bar
    g.close()
