"""Calls that the device has no room for: they fail with BO_ERR_OOM and leave the
simulator as it was.  The device is filled with one torch allocation for the call.

Bar: the same bits before and after."""
from __future__ import annotations

import contextlib

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


@contextlib.contextmanager
def _room(megabytes):
    """Leaves about this much free on the device."""
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - (megabytes << 20), dtype=torch.uint8,
                         device="cuda")
    try:
        yield
    finally:
        del filler
        torch.cuda.empty_cache()


def _factored(shape):
    from paper_1910_06059_gb300 import Sim
    m = synth.small_model(*shape, wells="5spot")
    g = Sim(m)
    g.set_state(*synth.random_state(m, seed_member=4))
    g.begin_step()
    g.assemble(2.0 * synth.DAY)
    g.factor()
    return g, np.random.default_rng(6).normal(size=3 * g.n)


def test_an_error_is_reported_once():
    """The one-CTA solve's factors (144 MB) do not fit; the next call on the thread
    succeeds."""
    from paper_1910_06059_gb300 import _lib
    g, r = _factored((60, 64, 64))
    z = g.precond_apply(r)
    g.solve_schedule = "block"
    with _room(64), pytest.raises(_lib.BoError, match="OOM"):
        g.precond_apply(r)
    g.solve_schedule = "tiled"
    assert np.array_equal(g.precond_apply(r), z)
    g.close()


@pytest.mark.parametrize("shape", [(60, 64, 64), (31, 41, 50)])
def test_mixed_precision_holds_its_factors_once(shape):
    """The FP32 factors (2 x 28 floats), D^-1 (9 doubles) and two FP32 vectors (4 floats) a
    slot of the 8 x 4-line tiles, and not the FP64 blocks (54 doubles) once more."""
    nx, ny, nz = shape
    g, r = _factored(shape)
    slots = 32 * -(-ny // 8) * -(-nz // 4) * (nx + 10)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    g.precision = "mixed"
    g.factor()
    g.precond_apply(r)
    torch.cuda.synchronize()
    held = before - torch.cuda.mem_get_info()[0]
    assert held <= slots * (4 * 56 + 8 * 9 + 2 * 4 * 4) + (12 << 20)
    g.close()


def test_mixed_precision_after_a_failed_switch():
    """The FP32 factors (64 MB) fit, the rest (30 MB) does not; a later switch gets it."""
    from paper_1910_06059_gb300 import _lib
    g, r = _factored((60, 64, 64))
    z = g.precond_apply(r)
    with _room(80), pytest.raises(_lib.BoError, match="OOM"):
        g.precision = "mixed"
    assert g.precision == "fp64" and np.array_equal(g.precond_apply(r), z)
    g.precision = "mixed"
    got = g.precond_apply(r)
    h, _ = _factored((60, 64, 64))
    h.precision = "mixed"
    assert np.array_equal(got, h.precond_apply(r))
    g.close()
    h.close()


def test_boxes_change_without_room_for_two_plans():
    """A sweep plan of this model takes 187 MB."""
    g, r = _factored((60, 64, 64))
    h, _ = _factored((60, 64, 64))
    h.subdomains, h.subdomains_z = 0, 12
    h.factor()
    want = h.precond_apply(r)
    h.close()
    with _room(100):
        g.subdomains_z = 12
        g.factor()
        assert np.array_equal(g.precond_apply(r), want)
    g.close()


def test_boxes_whose_plan_does_not_fit_leave_the_old_ones():
    """Boxes of 8 layers (3 + 3 + 2) take 14 MB more than one box."""
    from paper_1910_06059_gb300 import _lib
    g, r = _factored((60, 64, 64))
    z = g.precond_apply(r)
    with _room(4), pytest.raises(_lib.BoError, match="OOM"):
        g.subdomains_z = 8
    assert g.subdomains_z == 0
    g.factor()
    assert np.array_equal(g.precond_apply(r), z)
    g.subdomains_z = 8
    g.factor()
    assert not np.array_equal(g.precond_apply(r), z)
    g.close()
