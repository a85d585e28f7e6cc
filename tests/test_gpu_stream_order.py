"""Set-up calls of a simulator on a non-blocking stream while the legacy default stream
is busy: what such a call clears or uploads is ordered with the simulator's own work.

Bar: the same bits as with an idle device (each cell's value has one fixed order of
operations)."""
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


def _hold_legacy_stream():
    """About 50 ms of work on the legacy default stream."""
    torch.cuda._sleep(100_000_000)


# 16 x 14 tiles of 4 x 3 lines: more than one CTA per SM, so the grid differs between one
# and two
def _sim(stream, shape=(12, 64, 40)):
    from paper_1910_06059_gb300 import Sim
    m = synth.small_model(*shape, wells="5spot")
    g = Sim(m, stream=stream)
    g.set_state(*synth.random_state(m, seed_member=3))
    g.begin_step()
    g.assemble(2.0 * synth.DAY)
    return g


def _apply(g, r):
    g.factor()
    return g.precond_apply(r)


@pytest.mark.parametrize("call", ["ctas", "boxes"])
def test_sweep_setup_does_not_wait_for_the_legacy_stream(call):
    """A cleared ticket counter or plan that came late would be seen as wrong tiles."""
    st = torch.cuda.Stream()
    g = _sim(st)
    r = np.random.default_rng(5).normal(size=3 * g.n)

    def switch(on):
        if call == "ctas":
            g.set_sweep_ctas_per_sm(1 if on else 2)
        else:
            g.subdomains = 8 if on else 0

    switch(True)
    want_on = _apply(g, r)
    switch(False)
    want_off = _apply(g, r)
    for _ in range(3):
        _hold_legacy_stream()
        switch(True)
        on = _apply(g, r)
        _hold_legacy_stream()
        switch(False)
        off = _apply(g, r)
        assert np.array_equal(on, want_on) and np.array_equal(off, want_off)
    torch.cuda.synchronize()
    assert np.array_equal(_apply(g, r), want_off)
    g.close()
