"""Pointer walks on the longest chains: a stage whose walkers meet only
pointers as short as their own must not take time by the length of the chain.
Each test compares a stage with another of the same call or of a call on as
many edges without long chains, on the device's own clock."""
import pytest

from gpu_helpers import ctx

pytestmark = pytest.mark.gpu


def _stages(call, runs=3):
    """Smallest device time of every stage over some calls, after one more."""
    call()
    best = {}
    for _ in range(runs):
        call()
        for name, ms in ctx().stage_timing():
            best[name] = min(ms, best.get(name, ms))
    return best


def test_one_run_of_equal_weights():
    """One threshold: almost every merge has the same weight, so one run of
    tens of millions of merges collapses into its last. The collapse takes a
    few passes over the merges, as building the incidence lists does."""
    import torch
    E, V = 60_000_000, 3_000_000
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    src = torch.randint(0, V, (E,), generator=g, device="cuda")
    dst = (src + torch.randint(1, V, (E,), generator=g, device="cuda")) % V
    t = torch.randint(0, 30 * 86400, (E,), generator=g, device="cuda")
    src, dst = src.int(), dst.int()
    s = _stages(lambda: ctx().run_levels(src, dst, t, V, [1 << 20], 5))
    ctx().ws = None  # tens of GB: not kept for the tests after
    assert s["D2 condense and labels"] < 5 * s["A incidence lists"]
