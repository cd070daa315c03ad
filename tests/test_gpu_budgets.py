"""Budgets that hold a shape only without digit planes (program choice bit 3)."""
import pytest

from paper_1908_08553_gb300 import tn

pytestmark = pytest.mark.gpu


def _footprint(L, W, D, prec, knobs):
    probe = tn.tn_ctx_create(-1)
    lat = tn.tn_create_lattice(probe, L, W, D)
    try:
        tn.tn_autotune_set(L, W, D, prec, tn.TN_WORK_ENERGY, knobs)
        return tn.tn_footprint(lat, tn.TN_SCHED_AUTO, prec, tn.TN_WORK_ENERGY)
    finally:
        tn.tn_autotune_clear()
        tn.tn_destroy_lattice(lat)
        tn.tn_ctx_destroy(probe)


# by the context's budget, or by the caller's limit
@pytest.mark.parametrize("prec,L,W,D", [(tn.TN_FP64, 8, 8, 2), (tn.TN_FP32, 6, 6, 3)])
@pytest.mark.parametrize("by_budget", [True, False])
def test_autotuner_tunes_what_fits_without_planes(prec, L, W, D, by_budget):
    import torch
    torch.cuda.init()
    # the choices timed: the default, at D = 3 the one without bit 2 too
    codes = (15, 15 & ~4) if D == 3 else (15,)
    small = max(_footprint(L, W, D, prec, k & ~8) for k in codes)
    large = min(_footprint(L, W, D, prec, k) for k in codes)
    assert small < large
    ctx = tn.tn_ctx_create(0, small if by_budget else 0)
    try:
        tn.tn_autotune(ctx, [L], [W], [D], prec, reps=1, max_bytes=large if by_budget else small)
        got = tn.tn_autotune_lookup(L, W, D, prec)
        assert got["tuned"] and got["best_ms"] > 0.0
        assert got["knobs"] & 8         # where they fit, calls still take the digits
    finally:
        tn.tn_autotune_clear()
        tn.tn_ctx_destroy(ctx)
