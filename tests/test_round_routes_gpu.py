"""Rounds at a step's start go for all layers at once only where that is the shorter way: on both sides of the rules'
lines the launches are the expected ones, and the caches bit for bit the oracle's.  Scored rounds with a buffer that the
in-place compaction does not share between CTAs, and sets planned in the step whose plan takes the radix passes."""
import numpy as np
import pytest

from ra_testlib import Runner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,stacked", [(2, False), (3, True)], ids=["by-layer", "stacked"])
def test_scored_rounds_of_a_long_buffer(L, stacked):
    import paper_2609_03430_gb300 as ra

    K, r = 4096, 130
    run = Runner(L, 2, 2, [65], K, r, eseed=1, dseed=71, fused=True, policy=4)
    g = -(-4 * (K + 2 * r) // r) * r - 1  # the next step fires
    run.restore_full(g, layers=range(L))
    run.qsteps[0] = list(range(g))
    run.step_scale = [0.0] * g
    for l in range(L):
        w = run.up(np.stack([run.qrows(l, 0, s) for s in range(g - r, g)], axis=1)[None])
        ra.ra_restore_queries(run.ctx, l, w.data_ptr())
    ra.ra_profile_reset(run.ctx)
    run.step(check_attn_layers=(0, L - 1))
    select, stack = (ra.ra_profile_read(run.ctx, k)[1] for k in (ra.RA_KERNEL_SELECT, ra.RA_KERNEL_STACK))
    assert (select, stack) == ((1, 1) if stacked else (L, 0))
    run.step(check_attn_layers=(0, L - 1))
    run.check_state()
    run.close()


@pytest.mark.parametrize("L,planned", [(4, False), (16, True)], ids=["by-layer", "planned"])
def test_sets_of_a_long_buffer_planned_in_the_step(L, planned):
    import paper_2609_03430_gb300 as ra

    run = Runner(L, 2, 2, [33], 2000, 512, eseed=2, dseed=72, fused=True)
    run.restore_full(512 * 20 - 1, layers=range(L))
    ra.ra_profile_reset(run.ctx)
    run.step(check_attn_layers=(0, L - 1))
    evict, stack = (ra.ra_profile_read(run.ctx, k)[1] for k in (ra.RA_KERNEL_EVICT, ra.RA_KERNEL_STACK))
    assert (evict, stack) == ((0, 1) if planned else (L, 0))
    run.step(check_attn_layers=(0, L - 1))
    run.check_state()
    run.close()
