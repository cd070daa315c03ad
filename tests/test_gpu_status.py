"""A bounded device wait that gives up (its status word set from the host) is reported by
every call that runs contractions of its own."""
import numpy as np
import pytest

from paper_1908_08553_gb300 import inputs, tn

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    import torch
    torch.cuda.init()
    c = tn.tn_ctx_create(0, 0)
    yield c
    tn.tn_ctx_destroy(c)


# in one step: three norms (the first flagged), or three norms and the energy (all flagged)
@pytest.mark.parametrize("count,every", [(1, 0), (1, 1), (4, 1)])
def test_evolution_reports_a_timed_out_wait(ctx, count, every):
    L, W, D = 3, 4, 2
    A = inputs.random_lattice(L, W, D, 5300)
    lat = tn.tn_create_lattice(ctx, L, W, D)
    try:
        tn.tn_set_site_tensors(lat, A)
        tn.tn_ctx_inject_wait_timeout(ctx, count)
        with pytest.raises(tn.TNError) as e:
            tn.tn_ite_run(lat, L, W, 1.0, 3.04, 0.05, 1, D, 1e-12, every)
        assert e.value.status == tn.TN_ERR_TIMEOUT
        assert np.array_equal(tn.tn_get_site_tensors(lat, A.size), A)      # left as it was
        got = tn.tn_ite_run(lat, L, W, 1.0, 3.04, 0.05, 1, D, 1e-12, 1)[0]
        tn.tn_set_site_tensors(lat, A)
        assert np.array_equal(got, tn.tn_ite_run(lat, L, W, 1.0, 3.04, 0.05, 1, D, 1e-12, 1)[0])
    finally:
        tn.tn_destroy_lattice(lat)


def test_autotuner_reports_a_timed_out_wait(ctx):
    tn.tn_autotune_clear()
    try:
        for count in (1, 2):        # the warm-up; the warm-up and the timed run
            tn.tn_ctx_inject_wait_timeout(ctx, count)
            with pytest.raises(tn.TNError) as e:
                tn.tn_autotune(ctx, [4], [4], [2], tn.TN_FP64, reps=1)
            assert e.value.status == tn.TN_ERR_TIMEOUT
            tn.tn_ctx_inject_wait_timeout(ctx, 0)
        assert not tn.tn_autotune_lookup(4, 4, 2, tn.TN_FP64)["tuned"]
    finally:
        tn.tn_ctx_inject_wait_timeout(ctx, 0)
        tn.tn_autotune_clear()
