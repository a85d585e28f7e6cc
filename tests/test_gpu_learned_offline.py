"""Offline training of the learned stage under the settings that change how a kept
system's preconditioner is applied.

Every loss is ||u||^2 / ||r||^2 of one residual with the network unchanged (a learning
rate of 1e-30 moves no parameter), so a set has one mean loss whatever applies M^-1.
Bar: 1e-8 of it.  The schedules add the same products in other orders: 1e-16 of |A| |z|,
which is up to about 1e6 |r| in these systems, and a preconditioner of another system
moves the loss by far more."""
from __future__ import annotations

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

RTOL = 1e-8


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    from paper_1910_06059_gb300.build import build
    build()


def _collected(shape=(14, 18, 9), systems=4, before=None):
    """A simulator with a set of its own systems, collection off again."""
    from paper_1910_06059_gb300 import Sim
    g = Sim(synth.layered_model(*shape, config=1, name="layered"))
    if before:
        before(g)
    g.init_hydrostatic()
    g.learn_set_params(synth.learned_init(0))
    g.learn_collect(systems, samples=6)
    st, _ = g.step(2.0 * synth.DAY)
    assert st == 0
    g.learn_collect(0)
    assert g.learn_set_info()[0] == systems
    return g


def _loss(g):
    g.learn_set_params(synth.learned_init(0))
    first, last = g.learn_train_offline(epochs=2, lr=1e-30)
    assert np.isclose(first, last, rtol=1e-12)
    return first


def test_one_cta_schedule_trains_on_the_kept_systems():
    """Selected after the steps (nothing factorised since) and with another system's
    factors at hand."""
    g = _collected()
    want = _loss(g)
    g.solve_schedule = "block"
    assert np.isclose(_loss(g), want, rtol=RTOL)
    g.begin_step()
    g.assemble(30.0 * synth.DAY)
    g.factor()
    r = np.random.default_rng(2).normal(size=3 * g.n)
    z = g.precond_apply(r)
    assert np.isclose(_loss(g), want, rtol=RTOL)
    assert np.array_equal(g.precond_apply(r), z)      # the current factors are back
    st, _ = g.step(1.0 * synth.DAY)                   # another factorisation under it
    assert st == 0
    assert np.isclose(_loss(g), want, rtol=RTOL)
    g.solve_schedule = "tiled"
    assert np.isclose(_loss(g), want, rtol=1e-12)
    g.close()


def test_one_cta_schedule_holds_its_factors_only_where_it_runs():
    """A model that the one-CTA solve does not fit gathers nothing for it: no memory,
    no launch."""
    from paper_1910_06059_gb300 import Sim
    m = synth.small_model(20, 96, 48, wells="5spot")   # 144 tiles, 128 fit
    counts, free = [], []
    for schedule in ("tiled", "block"):
        g = Sim(m)
        g.set_state(*synth.random_state(m, seed_member=1))
        g.solve_schedule = schedule
        g.begin_step()
        g.assemble(2.0 * synth.DAY)
        torch.cuda.synchronize()
        before, launched = torch.cuda.mem_get_info()[0], g.launches
        g.factor()
        g.precond_apply(np.ones(3 * g.n))
        torch.cuda.synchronize()
        counts.append(g.launches - launched)
        free.append(before - torch.cuda.mem_get_info()[0])
        g.close()
    assert counts[0] == counts[1]
    assert free[1] <= free[0] + (8 << 20)   # the tile-order factors are 70 MB


def test_failed_training_leaves_the_current_factors():
    """The device has no room for the one-CTA solve's factors (144 MB), so the call fails
    on its first kept system; the factorisation made before still applies."""
    from paper_1910_06059_gb300 import _lib
    g = _collected((60, 64, 64), systems=1)
    g.begin_step()
    g.assemble(30.0 * synth.DAY)
    g.factor()
    r = np.random.default_rng(3).normal(size=3 * g.n)
    z = g.precond_apply(r)
    g.learn_set_params(synth.learned_init(0))
    g.solve_schedule = "block"
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - (64 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(_lib.BoError):
            g.learn_train_offline(epochs=1, lr=1e-30)
    finally:
        del filler
        torch.cuda.empty_cache()
    g.solve_schedule = "tiled"
    assert np.array_equal(g.precond_apply(r), z)
    g.solve_schedule = "block"
    first, _ = g.learn_train_offline(epochs=1, lr=1e-30)
    assert np.isfinite(first)
    g.close()


@pytest.mark.parametrize("boxes", [(0, 0), (16, 0), (0, 8), (16, 8)])
def test_kept_systems_keep_their_boxes(boxes):
    """A set collected with 8 x 4-line boxes has one preconditioner, whatever coarser
    boxes are set when it is trained on."""
    def narrow(g):
        g.subdomains, g.subdomains_z = 8, 4
    g = _collected((14, 21, 13), before=narrow)
    want = _loss(g)
    g.subdomains, g.subdomains_z = boxes
    assert np.isclose(_loss(g), want, rtol=RTOL)
    g.close()
